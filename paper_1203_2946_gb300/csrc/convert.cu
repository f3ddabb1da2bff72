// CRS <-> CMRS conversion kernels (Section 3; packing and the in-strip sort of
// Section 4) and their C-ABI entry points.
#include <algorithm>
#include <type_traits>

#include "common.cuh"

namespace cmrs {
namespace {

constexpr int kSortWarpCap = 1024;   // in-strip sort: strips up to this length (or less, see the launch) a warp each
constexpr int kSortBlockCap = 6144;  // up to this length a CTA each, longer ones by the radix sort
constexpr int kSortKeyedMin = 256, kSortKeyedCap = 1024;  // rows out of order: see k_sort_keyed
static_assert(kSortWarpCap <= kSortKeyedCap, "a strip that a warp lists has to fit k_sort_keyed's buffer");
constexpr int kSortWarps = 4;        // warps per CTA, a strip each
constexpr int kSortThreads = 256;    // threads sharing a strip of the CTA kernel
constexpr int kSortBatch = 4;        // independent loads each lane issues before using them
constexpr int kRadixThreads = 128;   // CTA radix sort for the longest strips
constexpr int kRadixWarps = kRadixThreads / 32;

struct StatusBlock {
  uint32_t status;
  int32_t max_strip;
  int32_t nblock, nradix, nkeyed;  // strips left to the CTA sort, to the radix sort, to the keyed sort
  uint32_t pad[59];
};

// ---------------------------------------------------------------- value forms
// F32: IEEE round to nearest even.  BF16: round to nearest even of the FP32
// value.  BF16X2: hi = BF16(v), lo = BF16(v - hi), the difference taken in
// double.  A float source skips the double: same bits, and no conversion on
// the FP64 pipe.
template <int DT>
struct Encode;
template <>
struct Encode<CMRS_F64> {
  typedef double Out;
  __device__ static void put(double v, Out *hi, Out *, int64_t k) { hi[k] = v; }
};
template <>
struct Encode<CMRS_F32> {
  typedef float Out;
  __device__ static void put(double v, Out *hi, Out *, int64_t k) { hi[k] = __double2float_rn(v); }
  // as through double and back: a signalling NaN comes out quiet, its other bits kept (no conversion: one on the
  // FP64 pipe costs its issue slot even where no lane needs it)
  __device__ static void put(float v, Out *hi, Out *, int64_t k) {
    if (v != v) v = __uint_as_float(__float_as_uint(v) | 0x00400000u);
    hi[k] = v;
  }
};
template <>
struct Encode<CMRS_BF16> {
  typedef uint16_t Out;
  __device__ static void put(double v, Out *hi, Out *, int64_t k) {
    put(__double2float_rn(v), hi, nullptr, k);
  }
  __device__ static void put(float v, Out *hi, Out *, int64_t k) {
    hi[k] = __bfloat16_as_ushort(__float2bfloat16_rn(v));
  }
};
template <>
struct Encode<CMRS_BF16X2> {
  typedef uint16_t Out;
  __device__ static void put(double v, Out *hi, Out *lo, int64_t k) {
    uint16_t h = __bfloat16_as_ushort(__float2bfloat16_rn(__double2float_rn(v)));
    double rest = __dsub_rn(v, (double)bf16_bits_to_float(h));
    hi[k] = h;
    lo[k] = __bfloat16_as_ushort(__float2bfloat16_rn(__double2float_rn(rest)));
  }
  // v - hi is a multiple of v's last place of at most 17 bits: FP32 holds it exactly
  __device__ static void put(float v, Out *hi, Out *lo, int64_t k) {
    const uint16_t h = __bfloat16_as_ushort(__float2bfloat16_rn(v));
    hi[k] = h;
    lo[k] = __bfloat16_as_ushort(__float2bfloat16_rn(__fsub_rn(v, bf16_bits_to_float(h))));
  }
};

// ---------------------------------------------------------------- packing
// The whole unsorted conversion in one pass.  A warp takes 32 consecutive rows
// at a time, row `lane`'s start in each lane.
//   Section 2.3: RowPtr[0] = 0, RowPtr[rows] = nnz, row lengths >= 0.  A group
// of rows with an invalid RowPtr range is flagged and skipped, so no access
// leaves the arrays.
//   Section 3: StripPtr[j] = RowPtr[j * height] for j < strips,
// StripPtr[strips] = nnz; the longest strip is recorded.
//   Section 4: packed = (col << bits) | (row mod height).  The rows' entries
// are one contiguous CRS range, walked with coalesced loads, kPackU batches of
// 32 in flight per lane.  The row of an entry is the number of row starts up
// to it: the starts that fall into a batch are joined into one 32-bit mask, so
// a batch costs one reduction and a bit count.  Where a group has empty rows
// (equal starts) an entry finds its row among the 32 starts by a five-step
// shuffle search instead.
// Bound by HBM: 67M FP32 entries (1.07 GB) in 174 us; with the search for every
// batch and a conversion through double for every value (the FP64 pipe 85%
// busy) it took 267 us, and the checks and StripPtr were two more launches.
constexpr int kPackU = 4;
template <typename In, int DT>
__global__ void k_pack(int rows, int cols, int nnz, int height, int strips, int bits,
                       const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ col_ind,
                       const In *__restrict__ val_in, int32_t *__restrict__ strip_ptr, uint32_t *__restrict__ packed,
                       typename Encode<DT>::Out *__restrict__ vhi, typename Encode<DT>::Out *__restrict__ vlo,
                       StatusBlock *st) {
  const unsigned kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int warps = (gridDim.x * blockDim.x) >> 5;
  const long long groups = ((long long)rows + 31) / 32;
  uint32_t bad = 0;
  int longest = 0;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    strip_ptr[strips] = nnz;
    if (row_ptr[0] != 0 || row_ptr[rows] != nnz) bad = ST_BAD_ROWPTR;
  }
  for (long long g = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; g < groups; g += warps) {
    const long long r0 = g * 32;
    const long long r = r0 + lane;
    // row `lane` of the group: [start, end); rows past the matrix are empty
    const int32_t start = r < rows ? row_ptr[r] : 0;
    const int32_t last = row_ptr[min(r0 + 32, (long long)rows)];
    int32_t end = __shfl_down_sync(kAll, start, 1);
    if (lane == 31 || r + 1 >= rows) end = last;
    const unsigned sj = (unsigned)r / (unsigned)height;  // r < rows + 32 fits 32 unsigned bits
    const int ris_r = (int)((unsigned)r - sj * (unsigned)height);
    if (r < rows && ris_r == 0) {
      strip_ptr[sj] = start;
      longest = max(longest, row_ptr[min(r + height, (long long)rows)] - start);
    }
    const bool ok = r >= rows || (start >= 0 && end >= start && end <= nnz);
    if (!__all_sync(kAll, ok)) {
      bad |= ST_BAD_ROWPTR;
      continue;
    }
    const int32_t e0 = __shfl_sync(kAll, start, 0);
    const int32_t e1 = last;
    const int nrows = (int)min(32LL, rows - r0);
    const int32_t key = lane < nrows ? start : e1;  // empty tail rows sort last
    const uint32_t ris_lane = (uint32_t)ris_r;
    const bool full = __all_sync(kAll, lane >= nrows || end > start);
    int before = -1;  // rows started before the batch, minus one
    for (int32_t k0 = e0; k0 < e1; k0 += 32 * kPackU) {
      int32_t c[kPackU];
      int j[kPackU];  // the row of the group holding the entry
      In v[kPackU];
#pragma unroll
      for (int u = 0; u < kPackU; ++u) {
        const int32_t k = k0 + 32 * u + lane;
        if (k < e1) {
          c[u] = col_ind[k];
          v[u] = val_in[k];
        }
      }
      if (full) {
#pragma unroll
        for (int u = 0; u < kPackU; ++u) {
          const int32_t kb = k0 + 32 * u;
          const unsigned rel = (unsigned)(key - kb);
          const unsigned starts = __reduce_or_sync(kAll, rel < 32u ? 1u << rel : 0u);
          j[u] = before + __popc(starts << (31 - lane));  // of which at or before this lane's entry
          before += __popc(starts);
        }
      } else {
#pragma unroll
        for (int u = 0; u < kPackU; ++u) {
          const int32_t k = k0 + 32 * u + lane;
          j[u] = 0;  // the last of the group's rows starting at or before k
#pragma unroll
          for (int step = 16; step >= 1; step >>= 1) {
            const int32_t s = __shfl_sync(kAll, key, j[u] + step);
            if (s <= k) j[u] += step;
          }
        }
      }
#pragma unroll
      for (int u = 0; u < kPackU; ++u) {
        const int32_t k = k0 + 32 * u + lane;
        const uint32_t ris = __shfl_sync(kAll, ris_lane, j[u]);
        if (k < e1) {
          int32_t col = c[u];
          if ((uint32_t)col >= (uint32_t)cols) {
            bad |= ST_BAD_COL;
            col = 0;
          }
          packed[k] = ((uint32_t)col << bits) | ris;
          Encode<DT>::put(v[u], vhi, vlo, k);
        }
      }
    }
  }
  bad = __reduce_or_sync(kAll, bad);
  longest = __reduce_max_sync(kAll, longest);
  if (lane == 0) {
    if (bad) atomicOr(&st->status, bad);
    if (longest > 0) atomicMax(&st->max_strip, longest);
  }
}

// ---------------------------------------------------------------- in-strip sort
// Section 4, fourth optimisation: each strip's entries ordered by column,
// ties kept in CRS order.  The sorted conversion reads the CRS arrays and
// writes the sorted strips directly: G threads (a warp, or a CTA for longer
// strips) take a strip, pack its words in shared memory, sort (word, position)
// pairs there and write words and values in order.
//   When the strip's rows are each already in column order (the usual CRS) the
// stable order is the order of the packed words -- equal columns differ in
// RowInStrip, which is CRS order -- and a merge tree over the rows sorts it:
// log2(height) rounds, each pair of runs shared by G / pairs threads, which
// split its output evenly (each finds its part by one binary search along the
// merge path) and merge it serially, without a branch.  A round costs about 15
// instructions per entry of a thread's share; the bitonic network below needs
// log2(n)^2 / 2 compare-exchanges per entry (20M entries, strips of 320 at
// height 16: 226 us, packing included, against 1,083 + 75).  Bound by
// instructions (178M, two thirds of them the merges) and shared-memory reads.
//   Otherwise the threads sort unique 64-bit keys (column << 32 | position in
// strip), which makes the order stable, with a bitonic network: strips of up to
// kSortKeyedMin entries where they are, longer ones up to kSortKeyedCap listed
// for k_sort_keyed, whose warps need half the buffer, and the rest by radix.
// (6M FP64 entries, rows shuffled: strips of 640, 1,280 and 4,800 entries 534,
// 617 and 454 us so, 821, 1,057 and 1,391 by the network in the merge's buffers.)
template <int G>
__device__ __forceinline__ void group_sync() {
  if constexpr (G == 32) __syncwarp();
  else __syncthreads();
}
template <int G>
__device__ __forceinline__ bool group_any(bool p) {
  if constexpr (G == 32) return __any_sync(0xffffffffu, p);
  else return __syncthreads_or(p);
}

// Row starts of strip s, row `lane` of it in each lane of every warp; false if
// its RowPtr range is invalid.
struct StripRows {
  int32_t start, end;  // row `lane`
  int32_t a, len;      // the strip's entries
  int nrow;
};
__device__ __forceinline__ bool strip_rows(int s, int rows, int nnz, int height, const int32_t *__restrict__ row_ptr,
                                           StripRows &R) {
  const unsigned kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int64_t r0 = (int64_t)s * height;
  R.nrow = (int)std::min<int64_t>(height, rows - r0);
  R.start = lane < R.nrow ? row_ptr[r0 + lane] : 0;
  const int32_t last = row_ptr[r0 + R.nrow];
  R.end = __shfl_down_sync(kAll, R.start, 1);
  if (lane == R.nrow - 1) R.end = last;
  R.a = __shfl_sync(kAll, R.start, 0);
  R.len = last - R.a;
  return __all_sync(kAll, lane >= R.nrow || (R.start >= 0 && R.end >= R.start && R.end <= nnz));
}

__device__ __forceinline__ uint32_t word_of(uint32_t v) { return v; }
__device__ __forceinline__ uint32_t word_of(uint2 v) { return v.x; }
__device__ __forceinline__ void make_entry(uint32_t word, uint32_t, uint32_t &v) { v = word; }
__device__ __forceinline__ void make_entry(uint32_t word, uint32_t pos, uint2 &v) { v = make_uint2(word, pos); }
__device__ __forceinline__ uint32_t pick(bool first, uint32_t a, uint32_t b) { return first ? a : b; }
__device__ __forceinline__ uint2 pick(bool first, uint2 a, uint2 b) {
  return make_uint2(first ? a.x : b.x, first ? a.y : b.y);
}

// Merge tree over the strip's rows, each in column order: log2(nrow) rounds of
// pairwise merges between src and dst (room for one entry more than the strip);
// returns the buffer that holds the result.
template <int G, typename E>
__device__ __forceinline__ E *merge_rows(E *src, E *dst, const int *rs, int nrow) {
  const int tid = G == 32 ? (int)(threadIdx.x & 31) : (int)threadIdx.x;
  for (int w = 1, lw = 0; w < nrow; w <<= 1, ++lw) {  // runs of w = 2^lw rows
    const int npairs = (nrow + 2 * w - 1) >> (lw + 1);
    const int ls = 31 - __clz(G) - (32 - __clz(npairs - 1));  // log2 of the threads per pair (__clz(0) = 32)
    const int share = 1 << ls, g = tid >> ls, t = tid & (share - 1);
    if (g < npairs) {
      const int b0 = rs[2 * w * g], b1 = rs[min(nrow, 2 * w * g + w)], b2 = rs[min(nrow, 2 * w * g + 2 * w)];
      const int n = ((b2 - b0 + share - 1) >> ls) | 1;  // odd: the threads' writes hit all banks
      const int d0 = min(t * n, b2 - b0), d1 = min(d0 + n, b2 - b0);
      int lo = max(0, d0 - (b2 - b1)), hi = min(d0, b1 - b0);
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (word_of(src[b0 + mid]) < word_of(src[b1 + d0 - 1 - mid])) lo = mid + 1;
        else hi = mid;
      }
      int ia = b0 + lo, ib = b1 + d0 - lo;
      E ka = src[ia], kb = src[ib];  // a read past a run's end goes unused
      for (int o = b0 + d0; o < b0 + d1; ++o) {
        const bool first = ia < b1 && (ib >= b2 || word_of(ka) < word_of(kb));
        dst[o] = pick(first, ka, kb);
        ia += first;
        ib += !first;
        const E v = src[first ? ia : ib];
        ka = pick(first, v, ka);
        kb = pick(first, kb, v);
      }
    }
    group_sync<G>();
    E *tmp = src;
    src = dst;
    dst = tmp;
  }
  return src;
}

// Unordered rows: n2 keys at `keys` (the power of two at or above len) from
// the packed words at `words`, sorted; key = column, row, position.
template <int G, typename E>
__device__ __forceinline__ void sort_keys(const E *words, unsigned long long *keys, int len, int bits) {
  const int tid = G == 32 ? (int)(threadIdx.x & 31) : (int)threadIdx.x;
  int n2 = 1;
  while (n2 < len) n2 <<= 1;
  // words and keys may overlap at the buffer's start: from the top down, G at
  // a time, a key never lands on a word still to be read
  for (int i0 = (n2 - 1) / G * G; i0 >= 0; i0 -= G) {
    const int i = i0 + tid;
    const uint32_t v = i < len ? word_of(words[i]) : 0u;
    group_sync<G>();
    if (i < n2)
      keys[i] = i < len ? ((unsigned long long)(v >> bits) << 32) | ((unsigned long long)(v & ((1u << bits) - 1)) << 16) |
                              (uint32_t)i
                        : ~0ull;
  }
  group_sync<G>();
  for (int k = 2; k <= n2; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = tid; i < n2; i += G) {
        const int ixj = i ^ j;
        if (ixj > i) {
          const unsigned long long u = keys[i], v = keys[ixj];
          const bool up = (i & k) == 0;
          if ((u > v) == up) {
            keys[i] = v;
            keys[ixj] = u;
          }
        }
      }
      group_sync<G>();
    }
  }
}

// One strip of at most cap entries by G threads; buf: 16 (cap + 1) bytes (kKeyed:
// 8 for each of the power of two at or above cap), rs: 33 words of shared memory.
// `bad`: a column was out of range (this thread's view).  Returns whether the
// strip was left alone, its rows out of order and more than `most` entries.
//   A warp merges the packed words alone: an entry's position in the strip is
// then its row's start plus its place among the row's entries, in sorted order
// as in CRS order, and its value waits in the other half of the buffer
// (copied there while the words are packed and merged).  A CTA merges (word,
// position) pairs and gathers the values from global memory.  kKeyed: no merge,
// the keys at once.
template <typename In, int DT, int G, bool kKeyed = false>
__device__ __forceinline__ bool sort_strip(const StripRows &R, int cols, int bits, int cap, int most, bool &bad,
                                           const int32_t *__restrict__ col_ind, const In *__restrict__ val_in,
                                           char *buf, int *rs, uint32_t *__restrict__ packed,
                                           typename Encode<DT>::Out *__restrict__ vhi,
                                           typename Encode<DT>::Out *__restrict__ vlo) {
  typedef typename std::conditional<G == 32, uint32_t, uint2>::type E;
  const unsigned kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int tid = G == 32 ? lane : (int)threadIdx.x;
  const int a = R.a, len = R.len, nrow = R.nrow;
  bool unordered = false;
  int32_t carry = 0;
  E *src = reinterpret_cast<E *>(buf), *dst = src + cap + 1;
  In *vals = reinterpret_cast<In *>(buf + 8 * ((size_t)cap + 1));  // the warp's values, behind both word buffers
  // row starts, relative to the strip
  if (tid < nrow) rs[tid] = R.start - a;
  if (tid == 0) rs[nrow] = len;
  if constexpr (G == 32 && !kKeyed) {
    for (int i = lane; i < len; i += 32)
      asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_u32(vals + i)), "l"(val_in + a + i),
                   "n"(sizeof(In))
                   : "memory");
  }
  // packed words
  const int32_t key = lane < nrow ? R.start : a + len;
  const bool full = __all_sync(kAll, lane >= nrow || R.end > R.start);
  for (int i0 = tid & ~31; i0 < len; i0 += G * kSortBatch) {
    int32_t c[kSortBatch], pc[kSortBatch];
#pragma unroll
    for (int u = 0; u < kSortBatch; ++u) {
      const int i = i0 + G * u + lane;
      c[u] = i < len ? col_ind[a + i] : 0;
      if (G > 32) pc[u] = lane == 0 && i > 0 && i < len ? col_ind[a + i - 1] : 0;
    }
#pragma unroll
    for (int u = 0; u < kSortBatch; ++u) {
      const int kb = a + i0 + G * u, k = kb + lane;
      if (kb >= a + len) break;  // warp-uniform
      int j = 0;                 // the row holding k: the last one starting at or before k
      bool first;                // whether k is its row's first entry
      if (full) {
        const unsigned rel = (unsigned)(key - kb);
        const unsigned starts = __reduce_or_sync(kAll, rel < 32u ? 1u << rel : 0u);
        j = __popc(__ballot_sync(kAll, key < kb)) - 1 + __popc(starts << (31 - lane));
        first = (starts >> lane) & 1u;
      } else {
#pragma unroll
        for (int step = 16; step >= 1; step >>= 1) {
          const int32_t sj = __shfl_sync(kAll, key, j + step);
          if (sj <= k) j += step;
        }
        first = __shfl_sync(kAll, key, j) == k;
      }
      int32_t prev = __shfl_sync(kAll, c[u], (lane + 31) & 31);  // lane 0: the chunk's last column, for the next chunk
      if (lane == 0) {
        const int32_t last = prev;
        prev = G > 32 ? pc[u] : carry;
        carry = last;
      }
      if (k < a + len) {
        if (!first && c[u] < prev) unordered = true;
        const bool out = (uint32_t)c[u] >= (uint32_t)cols;
        bad |= out;
        make_entry((out ? 0u : (uint32_t)c[u] << bits) | (uint32_t)j, (uint32_t)(k - a), src[k - a]);
      }
    }
  }
  const bool keyed = kKeyed || group_any<G>(unordered);
  group_sync<G>();
  if (keyed && len > most) {
    if constexpr (G == 32) asm volatile("cp.async.wait_all;" ::: "memory");
    group_sync<G>();  // the buffer is reused by the next strip
    return true;
  }
  unsigned long long *keys = reinterpret_cast<unsigned long long *>(buf);
  if (keyed) {
    if constexpr (G == 32) asm volatile("cp.async.wait_all;" ::: "memory");  // the keys take the whole buffer
    group_sync<G>();
    sort_keys<G>(src, keys, len, bits);
  } else if constexpr (!kKeyed) {
    src = merge_rows<G>(src, dst, rs, nrow);
  }
  const uint32_t mask = (1u << bits) - 1;
  if (!keyed && G == 32) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
    int next = lane < nrow ? rs[lane] : 0;
    with_row_bits(nrow, [&](auto nb) {
#pragma unroll 2
      for (int i0 = 0; i0 < len; i0 += 32) {
        const int i = i0 + lane;
        const uint32_t w = i < len ? word_of(src[i]) : 0u;
        const int at = place_in_row<decltype(nb)::value>((int)(w & mask), i < len, next);
        if (i < len) {
          packed[a + i] = w;
          Encode<DT>::put(vals[at], vhi, vlo, (int64_t)a + i);
        }
      }
    });
  } else {
    for (int i0 = tid; i0 < len; i0 += G * kSortBatch) {
      uint32_t w[kSortBatch];
      In x[kSortBatch];
#pragma unroll
      for (int u = 0; u < kSortBatch; ++u)
        if (i0 + G * u < len) {
          uint32_t pos;
          if (keyed) {
            const unsigned long long k = keys[i0 + G * u];
            w[u] = (uint32_t)((k >> 32) << bits) | (uint32_t)((k >> 16) & 0xffff);
            pos = (uint32_t)(k & 0xffff);
          } else {
            const uint2 *pairs = reinterpret_cast<const uint2 *>(src);  // a CTA's
            w[u] = pairs[i0 + G * u].x;
            pos = pairs[i0 + G * u].y;
          }
          x[u] = val_in[a + (int)pos];
        }
#pragma unroll
      for (int u = 0; u < kSortBatch; ++u)
        if (i0 + G * u < len) {
          packed[a + i0 + G * u] = w[u];
          Encode<DT>::put(x[u], vhi, vlo, (int64_t)a + i0 + G * u);
        }
    }
  }
  group_sync<G>();  // the buffer is reused by the next strip
  return false;
}

// Most strips of more than cap entries (cap >= 256) that do not overlap: with
// two lists of that length, one from either end, nnz words hold both.
__host__ __device__ __forceinline__ int list_room(int nnz, int cap) { return nnz / (cap + 1); }

// Validation, StripPtr and the longest strip as in k_pack; strips of up to cap
// entries sorted here (past kSortKeyedMin and out of order: listed for
// k_sort_keyed), longer ones listed for the kernels below: CTA strips from the
// front of the list, radix strips from its end, which the CTA sort adds its
// strips out of order to.  A strip is found valid by its own rows alone, so a
// RowPtr that falls back between strips makes many of them valid over the same
// entries; each list therefore ends after as many strips as can be that long
// without overlapping, and a ticket past it is an invalid RowPtr.
template <typename In, int DT>
__global__ void __launch_bounds__(kSortWarps * 32) k_sort_warp(int rows, int cols, int nnz, int height, int strips,
                                                               int bits, int cap, const int32_t *__restrict__ row_ptr,
                                                               const int32_t *__restrict__ col_ind,
                                                               const In *__restrict__ val_in,
                                                               int32_t *__restrict__ strip_ptr,
                                                               uint32_t *__restrict__ packed,
                                                               typename Encode<DT>::Out *__restrict__ vhi,
                                                               typename Encode<DT>::Out *__restrict__ vlo,
                                                               int32_t *__restrict__ list,
                                                               int32_t *__restrict__ keyed_list, StatusBlock *st) {
  extern __shared__ __align__(16) char smem[];
  __shared__ int rs_all[kSortWarps][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int room = list_room(nnz, cap);
  char *buf = smem + (size_t)w * 16 * (cap + 1);
  uint32_t bad = 0;
  int longest = 0;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    strip_ptr[strips] = nnz;
    if (row_ptr[0] != 0 || row_ptr[rows] != nnz) bad = ST_BAD_ROWPTR;
  }
  const int nw = gridDim.x * kSortWarps;
  for (int s = blockIdx.x * kSortWarps + w; s < strips; s += nw) {
    StripRows R;
    const bool ok = strip_rows(s, rows, nnz, height, row_ptr, R);
    if (lane == 0) strip_ptr[s] = R.a;
    if (!ok) {
      bad |= ST_BAD_ROWPTR;
      continue;
    }
    longest = max(longest, R.len);
    if (R.len > cap) {
      if (lane == 0) {
        const bool block = R.len <= kSortBlockCap;
        const int i = atomicAdd(block ? &st->nblock : &st->nradix, 1);
        if (i < room) list[block ? i : nnz - 1 - i] = s;
        else bad |= ST_BAD_ROWPTR;
      }
    } else if (R.len > 0) {
      bool bad_col = false;
      if (sort_strip<In, DT, 32>(R, cols, bits, cap, kSortKeyedMin, bad_col, col_ind, val_in, buf, rs_all[w], packed,
                                 vhi, vlo) &&
          lane == 0) {
        const int i = atomicAdd(&st->nkeyed, 1);
        if (i < list_room(nnz, kSortKeyedMin)) keyed_list[i] = s;
        else bad |= ST_BAD_ROWPTR;
      }
      if (bad_col) bad |= ST_BAD_COL;
    }
  }
  bad = __reduce_or_sync(0xffffffffu, bad);
  if (lane == 0) {
    if (bad) atomicOr(&st->status, bad);
    if (longest > 0) atomicMax(&st->max_strip, longest);
  }
}

// Listed strips of up to kSortBlockCap entries, a CTA each.  An invalid RowPtr
// (the status of k_sort_warp is complete here) leaves nothing to do: its lists
// were cut short and its strips may overlap.
template <typename In, int DT>
__global__ void __launch_bounds__(kSortThreads) k_sort_block(int rows, int cols, int nnz, int height, int bits,
                                                             const int32_t *__restrict__ row_ptr,
                                                             const int32_t *__restrict__ col_ind,
                                                             const In *__restrict__ val_in,
                                                             uint32_t *__restrict__ packed,
                                                             typename Encode<DT>::Out *__restrict__ vhi,
                                                             typename Encode<DT>::Out *__restrict__ vlo,
                                                             int32_t *list, int room, StatusBlock *st) {
  extern __shared__ __align__(16) char smem[];
  __shared__ int rs[33];
  if (st->status & ST_BAD_ROWPTR) return;
  const int n = st->nblock;
  bool bad = false;
  for (int i = blockIdx.x; i < n; i += gridDim.x) {
    StripRows R;
    const int s = list[i];
    strip_rows(s, rows, nnz, height, row_ptr, R);  // found valid when it was listed
    if (sort_strip<In, DT, kSortThreads>(R, cols, bits, kSortBlockCap, kSortKeyedCap, bad, col_ind, val_in, smem, rs,
                                         packed, vhi, vlo) &&
        threadIdx.x == 0) {
      const int k = atomicAdd(&st->nradix, 1);
      if (k < room) list[nnz - 1 - k] = s;  // always: the two lists' strips do not overlap
    }
  }
  if (bad) atomicOr(&st->status, ST_BAD_COL);
}

// Listed strips of kSortKeyedMin to kSortKeyedCap entries with rows out of
// order, a warp each, by keys alone: 8 bytes an entry of shared memory and none
// set aside for the longest strip's merge, 24 warps an SM where k_sort_warp's
// buffers of 1,024 entries leave 12.  6M FP64 entries in strips of 640,
// rows shuffled: 534 us for the whole conversion (821 in k_sort_warp).
template <typename In, int DT>
__global__ void __launch_bounds__(kSortWarps * 32) k_sort_keyed(int rows, int cols, int nnz, int height, int bits,
                                                                const int32_t *__restrict__ row_ptr,
                                                                const int32_t *__restrict__ col_ind,
                                                                const In *__restrict__ val_in,
                                                                uint32_t *__restrict__ packed,
                                                                typename Encode<DT>::Out *__restrict__ vhi,
                                                                typename Encode<DT>::Out *__restrict__ vlo,
                                                                const int32_t *__restrict__ list, const StatusBlock *st) {
  __shared__ __align__(16) char bufs[kSortWarps][8 * kSortKeyedCap];
  __shared__ int rs_all[kSortWarps][33];
  if (st->status & ST_BAD_ROWPTR) return;
  const int w = threadIdx.x >> 5, n = st->nkeyed, nw = gridDim.x * kSortWarps;
  bool bad = false;  // columns were checked when the strip was listed
  for (int i = blockIdx.x * kSortWarps + w; i < n; i += nw) {
    StripRows R;
    strip_rows(list[i], rows, nnz, height, row_ptr, R);
    sort_strip<In, DT, 32, true>(R, cols, bits, kSortKeyedCap, kSortKeyedCap, bad, col_ind, val_in, bufs[w], rs_all[w],
                                 packed, vhi, vlo);
  }
}

// The longest strips: one CTA per listed strip, stable
// least-significant-digit radix sort of (column, position) pairs through two
// global ping-pong buffers, 8 bits per pass.  Each pass: digit histogram,
// exclusive scan into bucket bases, then a stable scatter of 128-entry chunks
// ranked per warp with match_any and across warps by a per-digit prefix.
// Nothing is done with an invalid RowPtr: strips that overlap would share their
// part of the buffers.
template <typename In, int DT>
__global__ void __launch_bounds__(kRadixThreads) k_sort_radix(int rows, int cols, int nnz, int height, int bits,
                                                              int col_bits, const int32_t *__restrict__ row_ptr,
                                                              const int32_t *__restrict__ col_ind,
                                                              const In *__restrict__ val_in,
                                                              uint32_t *__restrict__ packed,
                                                              typename Encode<DT>::Out *__restrict__ vhi,
                                                              typename Encode<DT>::Out *__restrict__ vlo,
                                                              uint32_t *__restrict__ keyA, uint32_t *__restrict__ posA,
                                                              uint32_t *__restrict__ keyB, uint32_t *__restrict__ posB,
                                                              const int32_t *__restrict__ list, StatusBlock *st) {
  __shared__ int hist[256];
  __shared__ int base[256];
  __shared__ int ccount[256];
  __shared__ int wcnt[kRadixWarps][257];
  __shared__ int rs[33];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  if (st->status & ST_BAD_ROWPTR) return;
  const int nlist = st->nradix;
  bool bad = false;
  for (int li = blockIdx.x; li < nlist; li += gridDim.x) {
    StripRows R;
    strip_rows(list[nnz - 1 - li], rows, nnz, height, row_ptr, R);
    const int32_t a = R.a, len = R.len;
    if (tid < R.nrow) rs[tid] = R.start - a;
    for (int i = tid; i < len; i += kRadixThreads) {
      uint32_t c = (uint32_t)col_ind[a + i];
      if (c >= (uint32_t)cols) {
        bad = true;
        c = 0;
      }
      keyA[a + i] = c;
      posA[a + i] = (uint32_t)i;
    }
    uint32_t *ks = keyA, *ps = posA, *kd = keyB, *pd = posB;
    __syncthreads();
    for (int shift = 0; shift < col_bits; shift += 8) {
      for (int d = tid; d < 256; d += kRadixThreads) hist[d] = 0;
      for (int d = tid; d < kRadixWarps * 257; d += kRadixThreads) (&wcnt[0][0])[d] = 0;
      __syncthreads();
      for (int i = tid; i < len; i += kRadixThreads) atomicAdd(&hist[(ks[a + i] >> shift) & 255], 1);
      __syncthreads();
      if (tid == 0) {
        int run = 0;
        for (int d = 0; d < 256; ++d) {
          base[d] = run;
          run += hist[d];
        }
      }
      __syncthreads();
      for (int c0 = 0; c0 < len; c0 += kRadixThreads) {
        const int i = c0 + tid;
        const bool valid = i < len;
        uint32_t key = 0, pos = 0;
        int d = 256;
        if (valid) {
          key = ks[a + i];
          pos = ps[a + i];
          d = (key >> shift) & 255;
        }
        const uint32_t peers = __match_any_sync(0xffffffffu, d);
        const int rank = __popc(peers & ((1u << lane) - 1));
        if (valid && (__ffs(peers) - 1) == lane) wcnt[w][d] = __popc(peers);
        __syncthreads();
        for (int dd = tid; dd < 256; dd += kRadixThreads) {
          int run = 0;
          for (int ww = 0; ww < kRadixWarps; ++ww) {
            int t = wcnt[ww][dd];
            wcnt[ww][dd] = run;
            run += t;
          }
          ccount[dd] = run;
        }
        __syncthreads();
        if (valid) {
          int dst = base[d] + wcnt[w][d] + rank;
          kd[a + dst] = key;
          pd[a + dst] = pos;
        }
        __syncthreads();
        for (int dd = tid; dd < 256; dd += kRadixThreads) {
          base[dd] += ccount[dd];
          for (int ww = 0; ww < kRadixWarps; ++ww) wcnt[ww][dd] = 0;
        }
        __syncthreads();
      }
      uint32_t *t;
      t = ks; ks = kd; kd = t;
      t = ps; ps = pd; pd = t;
      __syncthreads();
    }
    for (int i = tid; i < len; i += kRadixThreads) {
      const int src = (int)ps[a + i];
      int j = 0;  // the row holding it: the last one starting at or before it
      for (int step = 16; step >= 1; step >>= 1)
        if (j + step < R.nrow && rs[j + step] <= src) j += step;
      packed[a + i] = (ks[a + i] << bits) | (uint32_t)j;
      Encode<DT>::put(val_in[a + src], vhi, vlo, (int64_t)a + i);
    }
    __syncthreads();
  }
  if (bad) atomicOr(&st->status, ST_BAD_COL);
}

// ---------------------------------------------------------------- CMRS -> CRS
// Sorted strips, one warp each: a stable counting sort by RowInStrip.  Its rows
// are counted; an exclusive scan over the rows gives RowPtr[s*h + r] =
// StripPtr[s] + #(RIS < r).  Staged (launch_to_csr says where): the strip's
// words are kept in shared memory on the way, then each chunk of 32 entries
// finds its places (place_in_row) and leaves its index there, so that columns
// and values go out coalesced, the values gathered from the strip's own range.
// Walked: a chunk of 32 entries after the other is read again, ranked by a
// match of its rows, and scattered to its places, one load round trip after
// another (20M FP64 entries in strips of 320: 275 us, staged 104 us).
//   Unsorted strips (kSorted false) already hold their entries in CRS order:
// the entry arrays are copied with the row bits dropped (coalesced, kPackU
// batches in flight per lane) and RowPtr[s*h + r] is the first entry of
// row r, found by a binary search of RowInStrip.
constexpr int kToCsrWarps = 8, kToCsrCap = 2048;  // most entries staged per warp
enum { T_PLAIN, T_STAGED, T_WALKED };  // unsorted strips; sorted ones, from the stage or from global memory
template <typename V, int kForm>
__global__ void __launch_bounds__(kToCsrWarps * 32) k_to_csr(
    int rows, int nnz, int height, int bits, int strips, int cap, const int32_t *__restrict__ sp,
    const uint32_t *__restrict__ packed, const V *__restrict__ vin, const V *__restrict__ vin_lo,
    int32_t *__restrict__ row_ptr, int32_t *__restrict__ col_out, V *__restrict__ vout, V *__restrict__ vout_lo,
    uint32_t *status) {
  extern __shared__ __align__(16) char smem[];
  __shared__ int cnt_all[kToCsrWarps][33];
  const unsigned kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int *cnt = cnt_all[w];
  uint32_t *words = reinterpret_cast<uint32_t *>(smem) + (size_t)w * cap;                        // T_STAGED: the strip
  uint16_t *from = reinterpret_cast<uint16_t *>(smem + (size_t)kToCsrWarps * cap * 4) + (size_t)w * cap;  // CRS order
  const uint32_t mask = (1u << bits) - 1;
  const int nw = gridDim.x * kToCsrWarps;
  uint32_t bad = 0;
  if (blockIdx.x == 0 && threadIdx.x == 0) row_ptr[rows] = nnz;
  for (int s = blockIdx.x * kToCsrWarps + w; s < strips; s += nw) {
    const int32_t a = sp[s], b = sp[s + 1];
    const int64_t row0 = (int64_t)s * height;
    const int nrow = (int)std::min<int64_t>(height, rows - row0);
    if (kForm == T_PLAIN) {
      int32_t start = a;
      if (lane > 0 && lane < nrow) {
        int32_t lo = a, hi = b;
        while (lo < hi) {
          const int32_t mid = lo + ((hi - lo) >> 1);
          if ((packed[mid] & mask) < (uint32_t)lane) lo = mid + 1;
          else hi = mid;
        }
        start = lo;
      }
      if (lane < nrow) row_ptr[row0 + lane] = start;
      for (int32_t i0 = a; i0 < b; i0 += 32 * kPackU) {
        uint32_t p[kPackU];
        V v[kPackU], vl[kPackU];
#pragma unroll
        for (int u = 0; u < kPackU; ++u) {
          const int32_t i = i0 + 32 * u + lane;
          if (i < b) {
            p[u] = packed[i];
            if (vout) {
              v[u] = vin[i];
              if (vout_lo) vl[u] = vin_lo[i];
            }
          }
        }
#pragma unroll
        for (int u = 0; u < kPackU; ++u) {
          const int32_t i = i0 + 32 * u + lane;
          if (i < b) {
            if ((p[u] & mask) >= (uint32_t)nrow) bad = 1;
            col_out[i] = (int32_t)(p[u] >> bits);
            if (vout) {
              vout[i] = v[u];
              if (vout_lo) vout_lo[i] = vl[u];
            }
          }
        }
      }
      continue;
    }
    cnt[lane] = 0;
    __syncwarp();
    const bool staged = kForm == T_STAGED && b - a <= cap;  // warp-uniform
    for (int32_t i0 = a; i0 < b; i0 += 32 * kPackU) {
      uint32_t p[kPackU];
#pragma unroll
      for (int u = 0; u < kPackU; ++u) {
        const int32_t i = i0 + 32 * u + lane;
        p[u] = i < b ? packed[i] : 0u;
      }
#pragma unroll
      for (int u = 0; u < kPackU; ++u) {
        const int32_t i = i0 + 32 * u + lane;
        if (i < b) {
          const int r = (int)(p[u] & mask);
          if (r >= nrow) bad = 1;
          else atomicAdd(&cnt[r], 1);
          if (staged) words[i - a] = p[u];
        }
      }
    }
    __syncwarp();
    int v = lane < nrow ? cnt[lane] : 0;
    int incl = v;
    for (int o = 1; o < 32; o <<= 1) {
      int t = __shfl_up_sync(kAll, incl, o);
      if (lane >= o) incl += t;
    }
    int next = a + incl - v;  // row `lane`'s next place
    if (lane < nrow) row_ptr[row0 + lane] = next;
    if (staged) {
      next -= a;
      with_row_bits(nrow, [&](auto nb) {
#pragma unroll 2
        for (int i0 = 0; i0 < b - a; i0 += 32) {
          const int i = i0 + lane;
          const int r = i < b - a ? (int)(words[i] & mask) : 0;
          const bool valid = i < b - a && r < nrow;
          const int at = place_in_row<decltype(nb)::value>(r, valid, next);
          if (valid) from[at] = (uint16_t)i;
        }
      });
      const int n = __shfl_sync(kAll, next, nrow - 1);  // entries placed
      __syncwarp();
      for (int i0 = 0; i0 < n; i0 += 32 * kPackU) {
        int f[kPackU];
        V x[kPackU], xl[kPackU];
#pragma unroll
        for (int u = 0; u < kPackU; ++u) {
          const int i = i0 + 32 * u + lane;
          if (i < n) {
            f[u] = from[i];
            if (vout) {
              x[u] = vin[a + f[u]];
              if (vout_lo) xl[u] = vin_lo[a + f[u]];
            }
          }
        }
#pragma unroll
        for (int u = 0; u < kPackU; ++u) {
          const int i = i0 + 32 * u + lane;
          if (i < n) {
            col_out[a + i] = (int32_t)(words[f[u]] >> bits);
            if (vout) {
              vout[a + i] = x[u];
              if (vout_lo) vout_lo[a + i] = xl[u];
            }
          }
        }
      }
      __syncwarp();  // the stage is reused by the next strip
      continue;
    }
    __syncwarp();
    cnt[lane] = next;  // running insertion point of row `lane`
    __syncwarp();
    for (int32_t i0 = a; i0 < b; i0 += 32) {
      const int32_t i = i0 + lane;
      int r = 32;
      uint32_t p = 0;
      if (i < b) {
        p = packed[i];
        r = (int)(p & mask);
        if (r >= nrow) r = 32;
      }
      const uint32_t peers = __match_any_sync(kAll, r);
      const int rank = __popc(peers & ((1u << lane) - 1));
      if (r < 32) {
        const int dst = cnt[r] + rank;
        col_out[dst] = (int32_t)(p >> bits);
        if (vout) {
          vout[dst] = vin[i];
          if (vout_lo) vout_lo[dst] = vin_lo[i];
        }
      }
      __syncwarp();
      if (r < 32 && (__ffs(peers) - 1) == lane) cnt[r] += __popc(peers);
      __syncwarp();
    }
    __syncwarp();
  }
  if (status && __any_sync(kAll, bad) && lane == 0) atomicOr(status, ST_BAD_RIS);
}

// ---------------------------------------------------------------- host glue
struct FromCsrLayout {
  size_t status = 0, list = 0, keyA = 0, posA = 0, keyB = 0, posB = 0, total = 0;
};

FromCsrLayout from_csr_layout(int nnz, int dtype, uint32_t flags) {
  FromCsrLayout L;
  size_t off = align256(sizeof(StatusBlock));
  if (flags & CMRS_SORTED) {
    L.list = off;  // two lists of list_room() strips
    off += align256((size_t)nnz * 4);
    L.keyA = off;
    off += align256((size_t)nnz * 4);
    L.posA = off;
    off += align256((size_t)nnz * 4);
    L.keyB = off;
    off += align256((size_t)nnz * 4);
    L.posB = off;
    off += align256((size_t)nnz * 4);
  }
  L.total = off;
  return L;
}

template <typename In, int DT>
int from_csr_impl(int rows, int cols, int nnz, int height, int bits, uint32_t flags, const int32_t *row_ptr,
                  const int32_t *col_ind, const In *val_in, int32_t *strip_ptr, uint32_t *packed, void *val_out,
                  char *ws, const FromCsrLayout &L, cudaStream_t st, int *max_strip) {
  typedef typename Encode<DT>::Out Out;
  StatusBlock *sb = reinterpret_cast<StatusBlock *>(ws + L.status);
  const int strips = (int)ceil_div(rows, height);
  CMRS_CUDA_TRY(cudaMemsetAsync(sb, 0, sizeof(StatusBlock), st));
  const int sms = sm_count();
  Out *vh = reinterpret_cast<Out *>(val_out);
  Out *vl = DT == CMRS_BF16X2 ? vh + cmrs_pad8(nnz) : nullptr;
  if (!(flags & CMRS_SORTED)) {
    int g = (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div((int64_t)rows, 256), (int64_t)sms * 16));  // 8 warps x 32 rows
    k_pack<In, DT><<<g, 256, 0, st>>>(rows, cols, nnz, height, strips, bits, row_ptr, col_ind, val_in, strip_ptr,
                                      packed, vh, vl, sb);
    CMRS_LAUNCH_CHECK();
  } else {
    int32_t *list = reinterpret_cast<int32_t *>(ws + L.list);
    int32_t *keyed = reinterpret_cast<int32_t *>(ws + L.keyB);  // read before the radix sort writes there
    // a warp's buffers: 1.5x an average strip and some, so that few strips go
    // to the CTA kernel and short ones leave shared memory for more warps
    const int64_t avg = strips > 0 ? nnz / strips : 0;
    const int cap = (int)std::min<int64_t>(kSortWarpCap, std::max<int64_t>(256, (avg + avg / 2 + 128) / 32 * 32));
    const size_t smem = (size_t)kSortWarps * 16 * (cap + 1);
    CMRS_CUDA_TRY(cudaFuncSetAttribute(k_sort_warp<In, DT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kSortWarps * 16 * (kSortWarpCap + 1)));
    int per_sm = 0;  // one resident wave: every warp walks the same number of strips
    CMRS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sort_warp<In, DT>, kSortWarps * 32, smem));
    int g = (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(strips, kSortWarps), (int64_t)sms * std::max(1, per_sm)));
    k_sort_warp<In, DT><<<g, kSortWarps * 32, smem, st>>>(rows, cols, nnz, height, strips, bits, cap, row_ptr, col_ind,
                                                          val_in, strip_ptr, packed, vh, vl, list, keyed, sb);
    CMRS_LAUNCH_CHECK();
    if (strips > 0 && nnz > cap) {  // a strip can be longer than that
      const int smem_b = 16 * (kSortBlockCap + 1);
      CMRS_CUDA_TRY(cudaFuncSetAttribute(k_sort_block<In, DT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_b));
      k_sort_block<In, DT><<<(int)std::min<int64_t>(strips, (int64_t)sms * 2), kSortThreads, smem_b, st>>>(
          rows, cols, nnz, height, bits, row_ptr, col_ind, val_in, packed, vh, vl, list, list_room(nnz, cap), sb);
      CMRS_LAUNCH_CHECK();
    }
    if (strips > 0 && nnz > kSortKeyedMin && cap > kSortKeyedMin) {
      k_sort_keyed<In, DT><<<(int)std::min<int64_t>(ceil_div(strips, kSortWarps), (int64_t)sms * 6), kSortWarps * 32, 0, st>>>(
          rows, cols, nnz, height, bits, row_ptr, col_ind, val_in, packed, vh, vl, keyed, sb);
      CMRS_LAUNCH_CHECK();
    }
    if (strips > 0 && nnz > kSortKeyedCap) {
      int col_bits = 1;
      while (col_bits < 31 && ((int64_t)1 << col_bits) < (int64_t)cols) ++col_bits;
      k_sort_radix<In, DT><<<(int)std::min<int64_t>(strips, (int64_t)sms * 4), kRadixThreads, 0, st>>>(
          rows, cols, nnz, height, bits, col_bits, row_ptr, col_ind, val_in, packed, vh, vl,
          reinterpret_cast<uint32_t *>(ws + L.keyA), reinterpret_cast<uint32_t *>(ws + L.posA),
          reinterpret_cast<uint32_t *>(ws + L.keyB), reinterpret_cast<uint32_t *>(ws + L.posB), list, sb);
      CMRS_LAUNCH_CHECK();
    }
  }
  StatusBlock host;
  CMRS_CUDA_TRY(cudaMemcpyAsync(&host, sb, 8, cudaMemcpyDeviceToHost, st));
  CMRS_CUDA_TRY(cudaStreamSynchronize(st));
  *max_strip = host.max_strip;
  if (host.status & (ST_BAD_ROWPTR | ST_BAD_COL)) return CMRS_ERR_CSR_INVALID;
  return CMRS_OK;
}

template <typename In>
int from_csr_dispatch(int dtype, int rows, int cols, int nnz, int height, int bits, uint32_t flags,
                      const int32_t *row_ptr, const int32_t *col_ind, const In *val_in, int32_t *strip_ptr,
                      uint32_t *packed, void *val_out, char *ws, const FromCsrLayout &L, cudaStream_t st,
                      int *max_strip) {
  switch (dtype) {
    case CMRS_F64:
      return from_csr_impl<In, CMRS_F64>(rows, cols, nnz, height, bits, flags, row_ptr, col_ind, val_in, strip_ptr,
                                         packed, val_out, ws, L, st, max_strip);
    case CMRS_F32:
      return from_csr_impl<In, CMRS_F32>(rows, cols, nnz, height, bits, flags, row_ptr, col_ind, val_in, strip_ptr,
                                         packed, val_out, ws, L, st, max_strip);
    case CMRS_BF16:
      return from_csr_impl<In, CMRS_BF16>(rows, cols, nnz, height, bits, flags, row_ptr, col_ind, val_in, strip_ptr,
                                          packed, val_out, ws, L, st, max_strip);
    case CMRS_BF16X2:
      return from_csr_impl<In, CMRS_BF16X2>(rows, cols, nnz, height, bits, flags, row_ptr, col_ind, val_in,
                                            strip_ptr, packed, val_out, ws, L, st, max_strip);
  }
  return CMRS_ERR_ARG;
}

}  // namespace
}  // namespace cmrs

using namespace cmrs;

extern "C" int cmrs_from_csr_workspace(int rows, int nnz, int height, uint32_t flags, int dtype, size_t *bytes) {
  if (!bytes || rows < 0 || nnz < 0 || dtype < CMRS_F64 || dtype > CMRS_BF16X2) return CMRS_ERR_ARG;
  if (cmrs_bits_for_height(height) < 0) return CMRS_ERR_HEIGHT;
  *bytes = from_csr_layout(nnz, dtype, flags).total;
  return CMRS_OK;
}

extern "C" int cmrs_from_csr(int rows, int cols, int nnz, const int32_t *row_ptr, const int32_t *col_ind,
                             const void *val_in, int val_in_dtype, int height, uint32_t flags, int dtype,
                             int32_t *strip_ptr_out, uint32_t *col_packed_out, void *val_out, void *workspace,
                             size_t workspace_bytes, void *stream, cmrs_matrix *out) {
  CMRS_TRACE();
  if (rows < 0 || cols < 0 || nnz < 0) return CMRS_ERR_ARG;
  if (dtype < CMRS_F64 || dtype > CMRS_BF16X2) return CMRS_ERR_ARG;
  if (val_in_dtype != CMRS_F64 && val_in_dtype != CMRS_F32) return CMRS_ERR_ARG;
  if (flags & ~CMRS_SORTED) return CMRS_ERR_ARG;
  const int bits = cmrs_bits_for_height(height);
  if (bits < 0) return CMRS_ERR_HEIGHT;
  if ((uint64_t)cols > ((uint64_t)1 << (32 - bits))) return CMRS_ERR_COL_OVERFLOW;
  if (!row_ptr || !strip_ptr_out) return CMRS_ERR_ARG;
  if (nnz > 0 && (!col_ind || !val_in || !col_packed_out || !val_out)) return CMRS_ERR_ARG;
  const FromCsrLayout L = from_csr_layout(nnz, dtype, flags);
  if (!workspace || workspace_bytes < L.total || (reinterpret_cast<uintptr_t>(workspace) & 255))
    return CMRS_ERR_WORKSPACE;
  int max_strip = 0;
  cudaStream_t st = as_stream(stream);
  char *ws = reinterpret_cast<char *>(workspace);
  int rc = val_in_dtype == CMRS_F64
               ? from_csr_dispatch<double>(dtype, rows, cols, nnz, height, bits, flags, row_ptr, col_ind,
                                           reinterpret_cast<const double *>(val_in), strip_ptr_out, col_packed_out,
                                           val_out, ws, L, st, &max_strip)
               : from_csr_dispatch<float>(dtype, rows, cols, nnz, height, bits, flags, row_ptr, col_ind,
                                          reinterpret_cast<const float *>(val_in), strip_ptr_out, col_packed_out,
                                          val_out, ws, L, st, &max_strip);
  if (rc != CMRS_OK) return rc;
  if (out) {
    out->rows = rows;
    out->cols = cols;
    out->nnz = nnz;
    out->height = height;
    out->strips = (int32_t)ceil_div(rows, height);
    out->bits = bits;
    out->flags = flags;
    out->dtype = dtype;
    out->max_strip_nnz = max_strip;
    out->strip_ptr = strip_ptr_out;
    out->col_packed = col_packed_out;
    out->val = val_out;
  }
  return CMRS_OK;
}

extern "C" int cmrs_to_csr_workspace(const cmrs_matrix *A, size_t *bytes) {
  if (!A || !bytes) return CMRS_ERR_ARG;
  *bytes = 256;
  return CMRS_OK;
}

template <typename V>
int launch_to_csr(bool sorted, cudaStream_t st, const cmrs_matrix *A, const V *vin, const V *vin_lo, int32_t *row_ptr,
                  int32_t *col_out, V *vout, V *vout_lo, uint32_t *status) {
  if (!sorted) {
    const int g = (int)std::min<int64_t>(ceil_div(A->strips, kToCsrWarps), (int64_t)sm_count() * 8);
    k_to_csr<V, T_PLAIN><<<g, kToCsrWarps * 32, 0, st>>>(A->rows, A->nnz, A->height, A->bits, A->strips, 0, A->strip_ptr,
                                                       A->col_packed, vin, vin_lo, row_ptr, col_out, vout, vout_lo,
                                                       status);
    return set_cuda_error(cudaGetLastError());
  }
  // stage: 1.5x an average strip, so that few strips are walked in global
  // memory and short ones leave room for more warps
  const int64_t avg = A->nnz / A->strips;
  const int cap = (int)std::min<int64_t>(kToCsrCap, (avg + avg / 2) / 32 * 32 + 64);
  // The stage pays where it saves a strip several load round trips and still
  // leaves warps to hide the rest (us walked -> staged, FP64): strips of 20, 40,
  // 80 entries 56 -> 105, 61 -> 94, 54 -> 58; of 160, 320, 640 76 -> 49, 92 ->
  // 46, 136 -> 67; of 2,000 and 2,500 91 -> 151, 105 -> 179.  Of few rows, long
  // strips scatter little (1,000 entries of one row 56 -> 60; of 8 rows 114 ->
  // 58), and 2-byte values less (160 entries of 4 rows 33 -> 38).  A strip far
  // past the stage is walked alone anyway, faster without one.
  const bool narrow = sizeof(V) == 2 && !vin_lo;
  const bool staged = avg >= 100 && avg <= std::min(1800, 600 * A->height) &&
                      (!narrow || A->height > 8 || (A->height == 8 && avg >= 200)) && A->max_strip_nnz <= 8 * cap;
  if (!staged) {
    const int g = (int)std::min<int64_t>(ceil_div(A->strips, kToCsrWarps), (int64_t)sm_count() * 8);
    k_to_csr<V, T_WALKED><<<g, kToCsrWarps * 32, 0, st>>>(A->rows, A->nnz, A->height, A->bits, A->strips, 0, A->strip_ptr,
                                                          A->col_packed, vin, vin_lo, row_ptr, col_out, vout, vout_lo,
                                                          status);
    return set_cuda_error(cudaGetLastError());
  }
  const size_t smem = (size_t)kToCsrWarps * cap * 6;
  CMRS_CUDA_TRY(cudaFuncSetAttribute(k_to_csr<V, T_STAGED>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     kToCsrWarps * kToCsrCap * 6));
  int per_sm = 0;
  CMRS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_to_csr<V, T_STAGED>, kToCsrWarps * 32, smem));
  const int g = (int)std::min<int64_t>(ceil_div(A->strips, kToCsrWarps), (int64_t)sm_count() * std::max(1, per_sm));
  k_to_csr<V, T_STAGED><<<g, kToCsrWarps * 32, smem, st>>>(A->rows, A->nnz, A->height, A->bits, A->strips, cap,
                                                       A->strip_ptr, A->col_packed, vin, vin_lo, row_ptr, col_out, vout,
                                                       vout_lo, status);
  return set_cuda_error(cudaGetLastError());
}

extern "C" int cmrs_to_csr(const cmrs_matrix *A, int32_t *row_ptr_out, int32_t *col_ind_out, void *val_out,
                           void *workspace, size_t workspace_bytes, void *stream) {
  CMRS_TRACE();
  if (!A || !row_ptr_out || A->rows < 0 || A->nnz < 0) return CMRS_ERR_ARG;
  if (cmrs_bits_for_height(A->height) != A->bits) return CMRS_ERR_HEIGHT;
  if (A->strips != ceil_div(A->rows, A->height)) return CMRS_ERR_ARG;
  if (A->nnz > 0 && (!A->col_packed || !col_ind_out || !A->strip_ptr)) return CMRS_ERR_ARG;
  if (A->dtype < CMRS_F64 || A->dtype > CMRS_BF16X2) return CMRS_ERR_ARG;
  if (A->flags & CMRS_PADDED) return CMRS_ERR_UNSUPPORTED;  // zero items are not told apart from entries
  uint32_t *status = (workspace && workspace_bytes >= 256) ? reinterpret_cast<uint32_t *>(workspace) : nullptr;
  cudaStream_t st = as_stream(stream);
  if (A->strips == 0) {
    CMRS_CUDA_TRY(cudaMemsetAsync(row_ptr_out, 0, sizeof(int32_t), st));
    return CMRS_OK;
  }
  const int64_t lo_off = cmrs_pad8(A->nnz);
  const bool sorted = (A->flags & CMRS_SORTED) != 0;
  switch (A->dtype) {
    case CMRS_F64:
      return launch_to_csr<double>(sorted, st, A, (const double *)A->val, nullptr, row_ptr_out, col_ind_out,
                            (double *)val_out, nullptr, status);
    case CMRS_F32:
      return launch_to_csr<float>(sorted, st, A, (const float *)A->val, nullptr, row_ptr_out, col_ind_out,
                           (float *)val_out, nullptr, status);
    case CMRS_BF16:
      return launch_to_csr<uint16_t>(sorted, st, A, (const uint16_t *)A->val, nullptr, row_ptr_out, col_ind_out,
                              (uint16_t *)val_out, nullptr, status);
    case CMRS_BF16X2:
      return launch_to_csr<uint16_t>(sorted, st, A, (const uint16_t *)A->val, (const uint16_t *)A->val + lo_off,
                              row_ptr_out, col_ind_out, (uint16_t *)val_out,
                              val_out ? (uint16_t *)val_out + lo_off : nullptr, status);
  }
  return CMRS_ERR_ARG;
}
