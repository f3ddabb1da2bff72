// A shared-memory stage of one contiguous range of a CMRS matrix's streams
// (packed words and values), filled by the bulk-copy engine.
#pragma once

#include "common.cuh"

namespace cmrs {

struct StageInfo {
  long long a8;
  int staged;
  int pad;
};

template <int DT>
struct Stage {
  typedef typename Form<DT>::Stored S;
  static constexpr bool kSplit = DT == CMRS_BF16X2;
  static constexpr size_t al(size_t b) { return (b + 127) & ~size_t(127); }
  static constexpr size_t colp_bytes(int cap) { return al((size_t)(cap + 8) * 4); }
  static constexpr size_t val_bytes(int cap) { return al((size_t)(cap + 8) * sizeof(S)); }
  static constexpr size_t bytes(int cap) { return colp_bytes(cap) + val_bytes(cap) * (kSplit ? 2 : 1); }
};

// One thread: copy entries [ea, eb) of the three streams into a stage.  The
// bulk copy covers the 8-entry-aligned body [a8, e8) (16-byte aligned for all
// forms); entries past the last full 8-group of the array are loaded by this
// thread, so nothing outside the arrays is read.
template <int DT>
__device__ void issue_stage(long long ea, long long eb, long long nnz, const uint32_t *packed,
                            const typename Form<DT>::Stored *hi, const typename Form<DT>::Stored *lo, char *stage,
                            int cap, uint64_t *bar, uint64_t pol, StageInfo *info) {
  typedef typename Form<DT>::Stored S;
  const long long a8 = ea & ~7LL, nnz8 = nnz & ~7LL;
  long long e8 = (eb + 7) & ~7LL;
  if (e8 > nnz8) e8 = nnz8;
  if (e8 < a8) e8 = a8;
  uint32_t *sc = reinterpret_cast<uint32_t *>(stage);
  S *sh = reinterpret_cast<S *>(stage + Stage<DT>::colp_bytes(cap));
  S *sl = reinterpret_cast<S *>(stage + Stage<DT>::colp_bytes(cap) + Stage<DT>::val_bytes(cap));
  for (long long k = e8; k < eb; ++k) {
    sc[k - a8] = packed[k];
    sh[k - a8] = hi[k];
    if (Stage<DT>::kSplit) sl[k - a8] = lo[k];
  }
  info->a8 = a8;
  info->staged = 1;
  const uint32_t cnt = (uint32_t)(e8 - a8);
  fence_proxy_async();
  mbar_arrive_expect_tx(bar, cnt * (4u + (uint32_t)sizeof(S) * (Stage<DT>::kSplit ? 2u : 1u)));
  if (cnt) {
    bulk_g2s(sc, packed + a8, cnt * 4u, bar, pol);
    bulk_g2s(sh, hi + a8, cnt * (uint32_t)sizeof(S), bar, pol);
    if (Stage<DT>::kSplit) bulk_g2s(sl, lo + a8, cnt * (uint32_t)sizeof(S), bar, pol);
  }
}

// One thread: copy words [ea, eb) of one 16-byte aligned array of n 32-bit
// words into dst (room for eb - ea + 8), word k at dst[k - (ea & ~3)].  As
// issue_stage: the bulk copy covers the 4-word-aligned body, the words past the
// array's last full group of four are loaded by this thread.
__device__ __forceinline__ void issue_words(int ea, int eb, int n, const int32_t *src, int32_t *dst, uint64_t *bar,
                                            uint64_t pol) {
  const int a4 = ea & ~3, n4 = n & ~3;
  const int e4 = max(a4, (int)min((long long)n4, ((long long)eb + 3) & ~3LL));
  for (int k = e4; k < eb; ++k) dst[k - a4] = src[k];
  fence_proxy_async();
  mbar_arrive_expect_tx(bar, (uint32_t)(e4 - a4) * 4u);
  if (e4 > a4) bulk_g2s(dst, src + a4, (uint32_t)(e4 - a4) * 4u, bar, pol);
}

}  // namespace cmrs
