// Strip selector: per-matrix features on the device, a small MLP (forward,
// backward, Adam) in FP32, and cmrs_select_strip.  Not in the paper: Section
// 6.2 picks the strip height by brute force over all heights and Section 6.7
// measures how much per-matrix tuning gains; here a network trained on this
// library's own timings predicts the choice, with the brute-force sweep as
// fallback and as the yardstick of its regret.
#include <algorithm>
#include <cmath>
#include <vector>

#include "common.cuh"
#include "stage.cuh"

namespace cmrs {
namespace {

constexpr int kNFeat = 32;
constexpr int kHeights[6] = {1, 2, 4, 8, 16, 32};
// choices 18, 19, 20: the modified CMRS of Section 6.6 at (height, slots)
constexpr int kPadChoice[3][2] = {{32, 1}, {32, 2}, {16, 8}};

struct FeatAcc {
  unsigned long long sum_l2, max_l, empty, same, near, sum_d, max_d;
  unsigned long long bins[8];
  unsigned long long spread[6], nonempty[6];
  // modified CMRS items at (32, 1), (32, 2), (16, 8); entries in rows of
  // >= 32, 512, 8192; sum of squares and max of 32-row strip entry counts
  unsigned long long pad[3], elong[3], s32_sq, s32_max;
  unsigned long long done;  // blocks finished
};

__device__ __forceinline__ unsigned long long warp_sum(unsigned long long v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// Features.  A warp takes 32 consecutive rows at a time, lane r row r: its
// bounds, its length statistics and its entries.  The rows' column indices are
// one contiguous range, which one bulk copy brings into the warp's
// shared-memory stage; each lane then walks its own row there, |col - row| and
// min / max in registers, no shuffle per entry (the furthest column of a row
// is its min or its max).  A range longer than the stage (or an array that is
// not 16-byte aligned) is read from global memory: a lane per row for rows of
// up to kFeatShort entries, the whole warp for longer ones.  The strips of
// every height h = 2^e <= 32 are aligned groups of h lanes, so a shuffle tree
// over the rows' min and max gives each strip's column spread in the same
// pass, and one over the row lengths each 32- and 16-row strip's entry count
// and longest row (the modified CMRS pass counts).  A group with an invalid
// RowPtr range is skipped.  The last block to finish computes the features, so
// there is no second launch.  16M entries in rows of 20..60: 41 us for all 32
// features; with one entry of the contiguous range per lane (an entry then
// finds its row by a five-step shuffle search and joins its row's min / max in
// a five-step scan: 69M warp instructions, here 17M) and a second kernel for
// the features, 153 us.  Reading the columns once is 10 us; what is left is
// each group's copy round trip and the walk's shared-memory reads.
constexpr int kFeatU = 4;        // loads in flight per lane
constexpr int kFeatShort = 64;   // unstaged rows up to this length: a lane each
constexpr int kFeatCap = 2048;   // most entries per stage
constexpr int kFeatThreads = 256;

// Entries first, first + step, ... of a row of len entries at c[0..]: whole
// batches of kFeatU without a guard, then one at a time.
__device__ __forceinline__ void feat_entries(const int32_t *__restrict__ c, unsigned first, unsigned step, unsigned len,
                                             int row, int &lo, int &hi, unsigned long long &sd, unsigned &near) {
  auto one = [&](int v) {
    // |v - row| of any two ints fits 32 unsigned bits
    const unsigned ad = (unsigned)max(v, row) - (unsigned)min(v, row);
    sd += ad;
    near += ad <= 64u;
    lo = min(lo, v);
    hi = max(hi, v);
  };
  unsigned k = first;
  for (; k + step * (kFeatU - 1) < len; k += step * kFeatU) {
    int v[kFeatU];
#pragma unroll
    for (int u = 0; u < kFeatU; ++u) v[u] = c[k + step * u];
#pragma unroll
    for (int u = 0; u < kFeatU; ++u) one(v[u]);
  }
  for (; k < len; k += step) one(c[k]);
}

// The features from the integer sums, with the same operations, in the same
// order, as their definition (no contraction into FMAs); thread t computes
// feature t.  Every division, root and logarithm is written once and shared by
// the features that need it: a branch per feature runs them one after another
// (20 us for the 32 features; FP64 issues one warp instruction in 16 cycles).
__device__ __forceinline__ void feat_final(int t, int rows, int nnz, const volatile FeatAcc *acc, double *f) {
  const double n = (double)rows, z = (double)nnz;
  const double ns = (double)((rows + 31) / 32);
  // mean row length; mean entries of a 32-row strip
  const double mean = __ddiv_rn(z, t >= 30 ? ns : n);
  const double mean1 = mean > 1.0 ? mean : 1.0;
  unsigned long long num = 0;
  double den = 1.0;  // dividing by 1 is exact
  bool plus1 = false, lg = false;
  if (t == 3) {
    num = acc->sum_l2;
    den = n;
  } else if (t == 4) {
    num = acc->max_l;
    plus1 = lg = true;
  } else if (t == 5) {
    num = acc->empty;
    den = n;
  } else if (t >= 6 && t < 14) {
    num = acc->bins[t - 6];
    den = n;
  } else if (t == 14) {
    if (nnz > 0) {
      num = acc->sum_d;
      den = z;
    }
    plus1 = lg = true;
  } else if (t == 15) {
    num = acc->max_d;
    plus1 = lg = true;
  } else if (t == 16) {
    if (nnz > 0) {
      num = acc->near;
      den = z;
    }
  } else if (t == 17) {
    if (rows > 1) {
      num = acc->same;
      den = (double)(rows - 1);
    }
  } else if (t >= 18 && t < 24) {
    const unsigned long long ne = acc->nonempty[t - 18];
    if (ne > 0) {
      num = acc->spread[t - 18];
      den = (double)ne;
    }
    plus1 = lg = true;
  } else if (t >= 24 && t < 27) {
    num = nnz > 0 ? acc->pad[t - 24] : 1ull;  // log2(1) = 0 for an empty matrix
    den = nnz > 0 ? z : 1.0;
    lg = true;
  } else if (t >= 27 && t < 30) {
    if (nnz > 0) {
      num = acc->elong[t - 27];
      den = z;
    }
  } else if (t == 30) {
    num = acc->s32_sq;
    den = ns;
  } else if (t == 31) {
    num = acc->s32_max;
    den = mean1;
    plus1 = lg = true;
  }
  double q = __ddiv_rn((double)num, den);
  if (t == 3 || t == 30) {  // spread of the lengths over their mean
    double var = __dsub_rn(q, __dmul_rn(mean, mean));
    if (var < 0.0) var = 0.0;
    q = __ddiv_rn(sqrt(var), mean1);
  }
  if (t == 0) q = n;
  if (t == 1) q = z > 1.0 ? z : 1.0;
  if (t == 2) q = mean;
  if (t == 2) plus1 = true;
  if (plus1) q = __dadd_rn(1.0, q);
  if (lg || t < 3) q = log2(q);
  f[t] = q;
}

__global__ void __launch_bounds__(kFeatThreads, 4) k_feat_rows(int rows, int nnz, int cap,
                                                               const int32_t *__restrict__ rp,
                                                               const int32_t *__restrict__ ci, FeatAcc *acc,
                                                               double *__restrict__ feat) {
  extern __shared__ __align__(128) char smem[];
  __shared__ uint64_t bars[kFeatThreads / 32];
  __shared__ unsigned long long s[35];
  __shared__ unsigned s_bins[9];  // rows by length: [2^q, 2^(q+1)) for q < 7, [128, ..), empty
  __shared__ bool s_last;
  for (int i = threadIdx.x; i < 35; i += kFeatThreads) s[i] = 0;
  if (threadIdx.x < 9) s_bins[threadIdx.x] = 0;
  const int w = threadIdx.x >> 5;
  int32_t *stg = reinterpret_cast<int32_t *>(smem) + (size_t)w * (cap + 8);
  if ((threadIdx.x & 31) == 0) {
    mbar_init(&bars[w], 1);
    fence_barrier_init();
  }
  __syncthreads();
  uint64_t pol = 0;
  if ((threadIdx.x & 31) == 0) pol = policy_evict_first();
  uint32_t phase = 0;
  bool stages = cap > 0;
  const unsigned kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const long long nw = ((long long)gridDim.x * kFeatThreads) >> 5;
  const long long groups = ((long long)rows + 31) / 32;
  unsigned long long l2 = 0, sd = 0, e32 = 0, e512 = 0, e8192 = 0, pad1 = 0, pad2 = 0, pad8 = 0, ssq = 0;
  unsigned long long spread[6] = {0, 0, 0, 0, 0, 0};
  unsigned mxl = 0, mxd = 0, smx = 0, same = 0, near = 0;  // counts of rows or entries: below 2^31
  unsigned nonempty = 0;                                   // lane e: strips of height 2^e with entries
  for (long long g = ((long long)blockIdx.x * kFeatThreads + threadIdx.x) >> 5; g < groups; g += nw) {
    const long long r0 = g * 32, r = r0 + lane;
    const int nrows = (int)min(32LL, (long long)rows - r0);
    const int start = r < rows ? rp[r] : 0;
    const int last = rp[min(r0 + 32, (long long)rows)];
    int end = __shfl_down_sync(kAll, start, 1);
    if (lane == 31 || r + 1 >= rows) end = last;
    const bool ok = lane >= nrows || (start >= 0 && end >= start && end <= nnz);
    if (!__all_sync(kAll, ok)) continue;
    const int e0 = __shfl_sync(kAll, start, 0);
    bool staged = stages && last > e0 && last - e0 <= cap;
    if (staged && lane == 0) issue_words(e0, last, nnz, ci, stg, &bars[w], pol);
    // row lengths (lane r)
    const int len = lane < nrows ? end - start : 0;
    int lprev = __shfl_up_sync(kAll, len, 1);
    if (lane == 0) lprev = r0 > 0 ? start - rp[r0 - 1] : -1;
    if (lane < nrows) {
      l2 += (unsigned long long)len * (unsigned)len;
      mxl = max(mxl, (unsigned)len);
      same += r > 0 && len == lprev;
      atomicAdd(&s_bins[len > 0 ? min(7, 31 - __clz(len)) : 8], 1u);
      e32 += len >= 32 ? len : 0;
      e512 += len >= 512 ? len : 0;
      e8192 += len >= 8192 ? len : 0;
    }
    // this group is strip g of height 32 and strips 2g, 2g+1 of height 16:
    // entries and longest row of each, by a shuffle tree over the lanes
    {
      unsigned ns = (unsigned)len, ms = ns;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        if (o == 16 && (lane & 15) == 0)  // the 16-row strips, before their halves meet
          pad8 += 32ull * max((ns + 31) / 32, (ms + 7) / 8);
        ns += __shfl_xor_sync(kAll, ns, o);
        ms = max(ms, __shfl_xor_sync(kAll, ms, o));
      }
      if (lane == 0) {
        pad1 += 32ull * ms;
        pad2 += 32ull * max((ns + 31) / 32, (ms + 1) / 2);
        ssq += (unsigned long long)ns * ns;
        smx = max(smx, ns);
      }
    }
    // entries: lo, hi become row `lane`'s min and max column
    int lo = INT32_MAX, hi = -1;
    if (staged) {
      if (__all_sync(kAll, mbar_wait_bounded(&bars[w], phase))) phase ^= 1;
      else staged = stages = false;  // read from global memory from here on; the late copy is waited for below
    }
    if (staged) {
      feat_entries(stg + (start - (e0 & ~3)), 0, 1, (unsigned)len, (int)r, lo, hi, sd, near);
      __syncwarp();  // every lane is done with the stage before the next copy lands in it
    } else {
      if (len <= kFeatShort) feat_entries(ci + start, 0, 1, (unsigned)len, (int)r, lo, hi, sd, near);
      for (unsigned m = __ballot_sync(kAll, len > kFeatShort); m; m &= m - 1) {
        const int src = __ffs(m) - 1;
        const int ks = __shfl_sync(kAll, start, src), kl = __shfl_sync(kAll, len, src);
        int a = INT32_MAX, b = -1;
        feat_entries(ci + ks, lane, 32, (unsigned)kl, (int)(r0 + src), a, b, sd, near);
        a = __reduce_min_sync(kAll, a);
        b = __reduce_max_sync(kAll, b);
        if (lane == src) {
          lo = a;
          hi = b;
        }
      }
    }
    if (len > 0)
      mxd = max(mxd, max((unsigned)max(hi, (int)r) - (unsigned)min(hi, (int)r),
                         (unsigned)max(lo, (int)r) - (unsigned)min(lo, (int)r)));
    // strip spreads: after step e each lane holds the min and max of its
    // aligned group of 2^e rows (rows past the matrix, and empty rows, are
    // neutral); the group's first lane counts the strip if it has entries
#pragma unroll
    for (int e = 0; e < 6; ++e) {
      if (e > 0) {
        lo = min(lo, __shfl_xor_sync(kAll, lo, 1 << (e - 1)));
        hi = max(hi, __shfl_xor_sync(kAll, hi, 1 << (e - 1)));
      }
      const bool counted = (lane & ((1 << e) - 1)) == 0 && hi >= 0;
      spread[e] += counted ? (unsigned)(hi - lo) : 0u;
      const unsigned c = __popc(__ballot_sync(kAll, counted));
      if (lane == e) nonempty += c;
    }
  }
  if (cap > 0 && !stages) mbar_wait_bounded(&bars[w], phase);
  // joined per warp, per block and over the blocks; the order does not matter
  auto add = [&](int i, unsigned long long v) {
    v = warp_sum(v);
    if (lane == 0 && v) atomicAdd(&s[i], v);
  };
  auto top = [&](int i, unsigned v) {
    v = __reduce_max_sync(kAll, v);
    if (lane == 0) atomicMax(&s[i], (unsigned long long)v);
  };
  add(0, l2);
  top(1, mxl);
  add(3, same);
  add(4, near);
  add(5, sd);
  top(6, mxd);
#pragma unroll
  for (int e = 0; e < 6; ++e) add(15 + e, spread[e]);
  if (lane < 6) atomicAdd(&s[21 + lane], (unsigned long long)nonempty);
  add(27, pad1);
  add(28, pad2);
  add(29, pad8);
  add(30, e32);
  add(31, e512);
  add(32, e8192);
  add(33, ssq);
  top(34, smx);
  __syncthreads();
  if (threadIdx.x < 9) s[threadIdx.x < 8 ? 7 + threadIdx.x : 2] = s_bins[threadIdx.x];
  __syncthreads();
  // s[] is laid out as FeatAcc's sums are
  unsigned long long *sums = reinterpret_cast<unsigned long long *>(acc);
  if (threadIdx.x < 35) {
    const unsigned long long v = s[threadIdx.x];
    if (threadIdx.x == 1 || threadIdx.x == 6 || threadIdx.x == 34) atomicMax(&sums[threadIdx.x], v);
    else if (v) atomicAdd(&sums[threadIdx.x], v);
    __threadfence();
  }
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(&acc->done, 1ull) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  if (threadIdx.x < kNFeat) feat_final(threadIdx.x, rows, nnz, acc, feat);
}

// ------------------------------------------------------------------ MLP (FP32)
// Z[n][j] = b[j] + sum_i W[j][i] X[n][i]; H = relu(Z) (or Z for the output).
__global__ void k_dense_fwd(int B, int nin, int nout, const float *__restrict__ X, const float *__restrict__ W,
                            const float *__restrict__ bias, float *__restrict__ Z, float *__restrict__ H, int relu) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= B * nout) return;
  const int n = t / nout, j = t - n * nout;
  float s = bias[j];
  for (int i = 0; i < nin; ++i) s = fmaf(W[j * nin + i], X[n * nin + i], s);
  if (Z) Z[t] = s;
  if (H) H[t] = relu ? fmaxf(s, 0.f) : s;
}

// gO = (O - T) / (B * nout)
__global__ void k_out_grad(int total, float scale, const float *__restrict__ O, const float *__restrict__ T,
                           float *__restrict__ G) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < total) G[i] = (O[i] - T[i]) * scale;
}

// All three layers' weight gradients in one launch: dW[j][i] = sum_n G[n][j]
// H[n][i], db[j] = sum_n G[n][j] (i == nin: H = 1), and the loss.  A block
// takes a tile of 32 inputs i (a lane each) by kGradJ outputs j of one layer;
// its warps take every kGradWarps-th sample, and their partial sums are added
// in warp order, so the sums do not depend on the launch.  With a thread
// walking the whole batch for one weight the three launches took 52 us at a
// batch of 256 (a chain of 256 dependent loads and FMAs, 60 blocks).
constexpr int kGradJ = 4, kGradWarps = 16;
struct GradLayer {
  int nin, nout;
  const float *G, *H;
  float *dW, *db;
};
struct GradArgs {
  GradLayer l[3];
  int tiles[3];  // blocks of each layer
};
__global__ void __launch_bounds__(kGradWarps * 32) k_weight_grads(int B, GradArgs ga, int nloss, float scale,
                                                                  const float *O,
                                                                  const float *T, float *loss) {
  __shared__ float part[kGradWarps][kGradJ][32];
  pdl_wait();
  pdl_launch_dependents();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int t = blockIdx.x, k = 0;
  while (k < 3 && t >= ga.tiles[k]) t -= ga.tiles[k++];
  if (k == 3) {  // the last block: loss = sum (O - T)^2 / (2 B nout), 256 partial sums joined by a tree
    float *p = &part[0][0][0];
    if (threadIdx.x < 256) {
      float s = 0.f;
      for (int i = threadIdx.x; i < nloss; i += 256) {
        const float e = O[i] - T[i];
        s = fmaf(e, e, s);
      }
      p[threadIdx.x] = s;
    }
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
      if ((int)threadIdx.x < h) p[threadIdx.x] += p[threadIdx.x + h];
      __syncthreads();
    }
    if (threadIdx.x == 0) *loss = 0.5f * p[0] * scale;
    return;
  }
  const GradLayer L = ga.l[k];
  const int itiles = L.nin / 32 + 1;  // nin + 1 inputs, the bias's 1 last
  const int i = (t % itiles) * 32 + lane, j0 = (t / itiles) * kGradJ;
  float s[kGradJ] = {};
#pragma unroll 8
  for (int n = w; n < B; n += kGradWarps) {
    const float h = i < L.nin ? L.H[(size_t)n * L.nin + i] : 1.f;
#pragma unroll
    for (int u = 0; u < kGradJ; ++u)
      if (j0 + u < L.nout) s[u] = fmaf(L.G[(size_t)n * L.nout + j0 + u], h, s[u]);
  }
#pragma unroll
  for (int u = 0; u < kGradJ; ++u) part[w][u][lane] = s[u];
  __syncthreads();
  if (w < kGradJ && j0 + w < L.nout && i <= L.nin) {
    float v = part[0][w][lane];
    for (int q = 1; q < kGradWarps; ++q) v += part[q][w][lane];
    if (i < L.nin) L.dW[(size_t)(j0 + w) * L.nin + i] = v;
    else L.db[j0 + w] = v;
  }
}

// These kernels start before the one ahead of them in the stream has ended and
// wait for it first thing (pdl_wait); none of their inputs is declared
// __restrict__, so that no read of it can be scheduled ahead of the wait.
//
// A block takes kMlpRows samples through all layers: the weights and the
// samples' activations are in shared memory, so a layer costs a block barrier
// instead of a launch and a trip through L2 (three launches, 15.7 us at a
// batch of 256).  A weight row is padded to an odd length: the lanes of a warp
// hold consecutive outputs j and read W[j][i] at the same i.  Every output is
// bias + one FMA chain over i, as k_dense_fwd sums it.  A training step at a
// batch of 256 (forward, backward, Adam): 98 us with ten launches, 39 us with
// these four, of which the host's launches and calls are most.
constexpr int kMlpRows = 4, kMlpThreads = 256;
constexpr size_t kMlpSmem = 96 * 1024;  // larger networks: a launch per layer
__host__ __device__ __forceinline__ int odd(int n) { return n | 1; }
__host__ __device__ __forceinline__ size_t mlp_smem_floats(int nin, int nh, int nout) {
  return (size_t)nh * odd(nin) + (size_t)nh * odd(nh) + (size_t)nout * odd(nh) + 2 * nh + nout +
         (size_t)kMlpRows * (nin + 2 * nh);
}
bool mlp_fits(int nin, int nh, int nout) { return mlp_smem_floats(nin, nh, nout) * 4 <= kMlpSmem; }

// `rows` rows of n floats into shared memory at a stride of ld floats, 4 bytes
// per cp.async (the padded rows allow no wider copy): all of a thread's words
// are in flight at once; mlp_copy_wait() before the block barrier.
__device__ __forceinline__ void mlp_copy(const float *src, float *dst, int rows, int n, int ld) {
  const int total = rows * n;
  const int dj = kMlpThreads / n, di = kMlpThreads - dj * n;  // a step of kMlpThreads words, in rows and columns
  int j = threadIdx.x / n, i = threadIdx.x - j * n;
  for (int t = threadIdx.x; t < total; t += kMlpThreads) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst + j * ld + i)), "l"(src + t) : "memory");
    j += dj;
    i += di;
    if (i >= n) {
      i -= n;
      ++j;
    }
  }
}
__device__ __forceinline__ void mlp_copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
// out(r, j, sum) for every sample r < R of the block and output j
template <typename F>
__device__ __forceinline__ void mlp_layer(int R, int nin, int nout, const float *W, const float *bias, const float *in,
                                          F out) {
  for (int t = threadIdx.x; t < R * nout; t += kMlpThreads) {
    const int r = t / nout, j = t - r * nout;
    const float *w = W + j * odd(nin), *x = in + r * nin;
    float s = bias[j];
#pragma unroll 8
    for (int i = 0; i < nin; ++i) s = fmaf(w[i], x[i], s);
    out(r, j, s);
  }
}
// The whole network on R samples held in x (shared), O(r, j, value) the outputs; Z1, H1, Z2, H2 (global, the block's
// first row) written when Z1 is not NULL.
template <typename F>
__device__ __forceinline__ void mlp_block(int R, int nin, int nh, int nout, const float *params,
                                          float *smem, float *Z1, float *H1, float *Z2, float *H2, F O) {
  float *W1 = smem, *W2 = W1 + nh * odd(nin), *W3 = W2 + nh * odd(nh), *b1 = W3 + nout * odd(nh), *b2 = b1 + nh,
        *b3 = b2 + nh, *x = b3 + nout, *a1 = x + kMlpRows * nin, *a2 = a1 + kMlpRows * nh;
  const float *p2 = params + nh * nin + nh, *p3 = p2 + nh * nh + nh;
  mlp_copy(params, W1, nh, nin, odd(nin));
  mlp_copy(p2, W2, nh, nh, odd(nh));
  mlp_copy(p3, W3, nout, nh, odd(nh));
  mlp_copy(params + nh * nin, b1, 1, nh, nh);
  mlp_copy(p2 + nh * nh, b2, 1, nh, nh);
  mlp_copy(p3 + nout * nh, b3, 1, nout, nout);
  mlp_copy_wait();
  __syncthreads();
  mlp_layer(R, nin, nh, W1, b1, x, [&](int r, int j, float s) {
    const float h = fmaxf(s, 0.f);
    a1[r * nh + j] = h;
    if (Z1) {
      Z1[r * nh + j] = s;
      H1[r * nh + j] = h;
    }
  });
  __syncthreads();
  mlp_layer(R, nh, nh, W2, b2, a1, [&](int r, int j, float s) {
    const float h = fmaxf(s, 0.f);
    a2[r * nh + j] = h;
    if (Z1) {
      Z2[r * nh + j] = s;
      H2[r * nh + j] = h;
    }
  });
  __syncthreads();
  mlp_layer(R, nh, nout, W3, b3, a2, O);
}
__device__ __forceinline__ float *mlp_x(float *smem, int nin, int nh, int nout) {
  return smem + nh * odd(nin) + nh * odd(nh) + nout * odd(nh) + 2 * nh + nout;
}

__global__ void __launch_bounds__(kMlpThreads) k_mlp_fwd(int B, int nin, int nh, int nout, const float *X,
                                                         const float *params, float *Z1, float *H1,
                                                         float *Z2, float *H2, float *O) {
  extern __shared__ float smem_f[];
  pdl_wait();
  pdl_launch_dependents();
  const size_t n0 = (size_t)blockIdx.x * kMlpRows;
  const int R = (int)min((size_t)kMlpRows, (size_t)B - n0);
  float *x = mlp_x(smem_f, nin, nh, nout);
  for (int t = threadIdx.x; t < R * nin; t += kMlpThreads) x[t] = X[n0 * nin + t];
  const size_t at = n0 * nh;
  mlp_block(R, nin, nh, nout, params, smem_f, Z1 + at, H1 + at, Z2 + at, H2 + at,
            [&](int r, int j, float s) { O[(n0 + r) * nout + j] = s; });
}

// Backward through the samples: gO = (O - T) / (B nout), g2 = (Z2 > 0) W3^T gO,
// g1 = (Z1 > 0) W2^T g2, kMlpRows samples per block, W2 and W3 in shared
// memory.
__host__ __device__ __forceinline__ size_t mlp_bwd_smem_floats(int nh, int nout) {
  return (size_t)nh * nh + (size_t)nout * nh + (size_t)kMlpRows * (nout + nh);
}
__global__ void __launch_bounds__(kMlpThreads) k_mlp_bwd(int B, int nh, int nout, float scale, const float *O,
                                                         const float *T, const float *W2, const float *W3,
                                                         const float *Z1, const float *Z2, float *gO, float *g2,
                                                         float *g1) {
  extern __shared__ float smem_f[];
  pdl_wait();
  pdl_launch_dependents();
  const size_t n0 = (size_t)blockIdx.x * kMlpRows;
  const int R = (int)min((size_t)kMlpRows, (size_t)B - n0);
  float *w2 = smem_f, *w3 = w2 + nh * nh, *so = w3 + nout * nh, *s2 = so + kMlpRows * nout;
  mlp_copy(W3, w3, nout, nh, nh);
  mlp_copy(W2, w2, nh, nh, nh);
  for (int t = threadIdx.x; t < R * nout; t += kMlpThreads) {
    const float g = (O[n0 * nout + t] - T[n0 * nout + t]) * scale;
    so[t] = g;
    gO[n0 * nout + t] = g;
  }
  mlp_copy_wait();
  __syncthreads();
  for (int t = threadIdx.x; t < R * nh; t += kMlpThreads) {
    const int r = t / nh, i = t - r * nh;
    const float z = Z2[n0 * nh + t];
    float s = 0.f;
#pragma unroll 8
    for (int j = 0; j < nout; ++j) s = fmaf(w3[j * nh + i], so[r * nout + j], s);
    s = z > 0.f ? s : 0.f;
    s2[t] = s;
    g2[n0 * nh + t] = s;
  }
  __syncthreads();
  for (int t = threadIdx.x; t < R * nh; t += kMlpThreads) {
    const int r = t / nh, i = t - r * nh;
    const float z = Z1[n0 * nh + t];
    float s = 0.f;
#pragma unroll 8
    for (int j = 0; j < nh; ++j) s = fmaf(w2[j * nh + i], s2[r * nh + j], s);
    g1[n0 * nh + t] = z > 0.f ? s : 0.f;
  }
}

// Gin[n][i] = (Z[n][i] > 0) * sum_j W[j][i] G[n][j]
__global__ void k_back_hidden(int B, int nin, int nout, const float *__restrict__ G, const float *__restrict__ W,
                              const float *__restrict__ Z, float *__restrict__ Gin) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= B * nin) return;
  const int n = t / nin, i = t - n * nin;
  float s = 0.f;
  for (int j = 0; j < nout; ++j) s = fmaf(W[j * nin + i], G[n * nout + j], s);
  Gin[t] = Z[t] > 0.f ? s : 0.f;
}

// Adam (Kingma and Ba 2015); c1 = 1 - beta1^t, c2 = 1 - beta2^t.
__global__ void k_adam(int n, float *p, const float *g, float *m,
                       float *v, float lr, float b1, float b2, float eps, float c1, float c2) {
  pdl_wait();
  pdl_launch_dependents();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// One matrix through the selector, one block: x = (f - mean) * scale as FP32
// network input, the network, and the argmin of its predicted cost over the
// choices (the first of equal costs).
__global__ void __launch_bounds__(kMlpThreads) k_choose(int nin, int nh, int nout, const double *f,
                                                        const float *mean,
                                                        const float *scale,
                                                        const float *params, int *out) {
  extern __shared__ float smem_f[];
  __shared__ float cost[CMRS_SEL_CHOICES];
  float *x = mlp_x(smem_f, nin, nh, nout);
  pdl_wait();
  pdl_launch_dependents();
  for (int i = threadIdx.x; i < nin; i += kMlpThreads) x[i] = ((float)f[i] - mean[i]) * scale[i];
  mlp_block(1, nin, nh, nout, params, smem_f, nullptr, nullptr, nullptr, nullptr,
            [&](int, int j, float s) { cost[j] = s; });
  __syncthreads();
  if (threadIdx.x != 0) return;
  int best = 0;
  for (int i = 1; i < nout; ++i)
    if (cost[i] < cost[best]) best = i;
  *out = best;
}

inline int grid_for(long long n, int t) { return (int)std::max<long long>(1, (n + t - 1) / t); }

size_t param_count(int nin, int nh, int nout) {
  return (size_t)nh * nin + nh + (size_t)nh * nh + nh + (size_t)nout * nh + nout;
}

size_t features_ws(int rows) {
  (void)rows;
  return align256(sizeof(FeatAcc));
}

}  // namespace
}  // namespace cmrs

using namespace cmrs;

extern "C" int cmrs_features_workspace(int rows, size_t *bytes) {
  if (rows < 0 || !bytes) return CMRS_ERR_ARG;
  *bytes = features_ws(rows);
  return CMRS_OK;
}

extern "C" int cmrs_features(int rows, int nnz, const int32_t *row_ptr, const int32_t *col_ind, double *feat,
                             void *workspace, size_t workspace_bytes, void *stream) {
  CMRS_TRACE();
  if (rows < 1 || nnz < 0 || !row_ptr || !feat || (nnz > 0 && !col_ind)) return CMRS_ERR_ARG;
  if (!workspace || workspace_bytes < features_ws(rows) || (reinterpret_cast<uintptr_t>(workspace) & 255))
    return CMRS_ERR_WORKSPACE;
  cudaStream_t st = as_stream(stream);
  char *ws = reinterpret_cast<char *>(workspace);
  FeatAcc *acc = reinterpret_cast<FeatAcc *>(ws);
  CMRS_CUDA_TRY(cudaMemsetAsync(acc, 0, sizeof(FeatAcc), st));
  const int sms = sm_count();
  // stage: 1.25x an average group's entries, so that most groups fit and short
  // rows leave shared memory for more warps; none where bulk copies cannot go
  const long long avg = 32LL * nnz / rows;
  const int cap = (reinterpret_cast<uintptr_t>(col_ind) & 15) == 0 && nnz > 0
                      ? (int)std::min<long long>(kFeatCap, (avg + avg / 4) / 32 * 32 + 64)
                      : 0;
  const size_t smem = cap ? (size_t)(kFeatThreads / 32) * (cap + 8) * 4 : 0;
  const int g = (int)std::min<long long>(ceil_div((long long)rows, kFeatThreads), (long long)sms * 4);
  CMRS_CUDA_TRY(cudaFuncSetAttribute(k_feat_rows, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)((kFeatThreads / 32) * (kFeatCap + 8) * 4)));
  k_feat_rows<<<g, kFeatThreads, smem, st>>>(rows, nnz, cap, row_ptr, col_ind, acc, feat);
  CMRS_LAUNCH_CHECK();
  return CMRS_OK;
}

extern "C" int64_t cmrs_mlp_param_count(int nin, int nh, int nout) {
  if (nin < 1 || nh < 1 || nout < 1) return -1;
  return (int64_t)param_count(nin, nh, nout);
}

// acts layout: Z1[B][nh], H1[B][nh], Z2[B][nh], H2[B][nh], O[B][nout]
extern "C" int cmrs_mlp_forward(int B, int nin, int nh, int nout, const float *X, const float *params, float *acts,
                                void *stream) {
  CMRS_TRACE();
  if (B < 1 || nin < 1 || nh < 1 || nout < 1 || !X || !params || !acts) return CMRS_ERR_ARG;
  cudaStream_t st = as_stream(stream);
  const float *W1 = params, *b1 = W1 + (size_t)nh * nin, *W2 = b1 + nh, *b2 = W2 + (size_t)nh * nh, *W3 = b2 + nh,
              *b3 = W3 + (size_t)nout * nh;
  float *Z1 = acts, *H1 = Z1 + (size_t)B * nh, *Z2 = H1 + (size_t)B * nh, *H2 = Z2 + (size_t)B * nh,
        *O = H2 + (size_t)B * nh;
  if (mlp_fits(nin, nh, nout)) {
    const size_t smem = mlp_smem_floats(nin, nh, nout) * 4;
    if (smem > 48 * 1024)
      CMRS_CUDA_TRY(cudaFuncSetAttribute(k_mlp_fwd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMlpSmem));
    return launch_pdl(k_mlp_fwd, (unsigned)ceil_div(B, kMlpRows), kMlpThreads, smem, st, B, nin, nh, nout, X, params, Z1,
                      H1, Z2, H2, O);
  }
  k_dense_fwd<<<grid_for((long long)B * nh, 128), 128, 0, st>>>(B, nin, nh, X, W1, b1, Z1, H1, 1);
  k_dense_fwd<<<grid_for((long long)B * nh, 128), 128, 0, st>>>(B, nh, nh, H1, W2, b2, Z2, H2, 1);
  k_dense_fwd<<<grid_for((long long)B * nout, 128), 128, 0, st>>>(B, nh, nout, H2, W3, b3, nullptr, O, 0);
  CMRS_LAUNCH_CHECK();
  return CMRS_OK;
}

// Loss 1/(2 B nout) sum (O - T)^2 and its gradient (same layout as params).
// scratch: B * (nout + 2 nh) floats.  loss: device float (may be NULL).
extern "C" int cmrs_mlp_backward(int B, int nin, int nh, int nout, const float *X, const float *T,
                                 const float *params, const float *acts, float *grads, float *scratch, float *loss,
                                 void *stream) {
  CMRS_TRACE();
  if (B < 1 || nin < 1 || nh < 1 || nout < 1 || !X || !T || !params || !acts || !grads || !scratch)
    return CMRS_ERR_ARG;
  cudaStream_t st = as_stream(stream);
  const float *W2 = params + (size_t)nh * nin + nh, *W3 = W2 + (size_t)nh * nh + nh;
  const float *Z1 = acts, *H1 = Z1 + (size_t)B * nh, *Z2 = H1 + (size_t)B * nh, *H2 = Z2 + (size_t)B * nh,
              *O = H2 + (size_t)B * nh;
  float *dW1 = grads, *db1 = dW1 + (size_t)nh * nin, *dW2 = db1 + nh, *db2 = dW2 + (size_t)nh * nh,
        *dW3 = db2 + nh, *db3 = dW3 + (size_t)nout * nh;
  float *gO = scratch, *g2 = gO + (size_t)B * nout, *g1 = g2 + (size_t)B * nh;
  const float scale = 1.0f / ((float)B * (float)nout);
  const size_t smem = mlp_bwd_smem_floats(nh, nout) * 4;
  if (smem <= kMlpSmem) {
    if (smem > 48 * 1024)
      CMRS_CUDA_TRY(cudaFuncSetAttribute(k_mlp_bwd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMlpSmem));
    const int rc = launch_pdl(k_mlp_bwd, (unsigned)ceil_div(B, kMlpRows), kMlpThreads, smem, st, B, nh, nout, scale, O,
                              T, W2, W3, Z1, Z2, gO, g2, g1);
    if (rc) return rc;
  } else {  // wide layers: a launch per layer
    k_out_grad<<<grid_for((long long)B * nout, 256), 256, 0, st>>>(B * nout, scale, O, T, gO);
    k_back_hidden<<<grid_for((long long)B * nh, 128), 128, 0, st>>>(B, nh, nout, gO, W3, Z2, g2);
    k_back_hidden<<<grid_for((long long)B * nh, 128), 128, 0, st>>>(B, nh, nh, g2, W2, Z1, g1);
    CMRS_LAUNCH_CHECK();
  }
  GradArgs ga;
  ga.l[0] = GradLayer{nh, nout, gO, H2, dW3, db3};
  ga.l[1] = GradLayer{nh, nh, g2, H1, dW2, db2};
  ga.l[2] = GradLayer{nin, nh, g1, X, dW1, db1};
  int blocks = 0;
  for (int k = 0; k < 3; ++k) {
    ga.tiles[k] = (ga.l[k].nin / 32 + 1) * (int)ceil_div(ga.l[k].nout, kGradJ);
    blocks += ga.tiles[k];
  }
  return launch_pdl(k_weight_grads, (unsigned)(blocks + (loss ? 1 : 0)), kGradWarps * 32, 0, st, B, ga, B * nout, scale,
                    O, T, loss);
}

extern "C" int cmrs_mlp_adam(int n, float *params, const float *grads, float *m, float *v, int step, float lr,
                             float beta1, float beta2, float eps, void *stream) {
  CMRS_TRACE();
  if (n < 1 || !params || !grads || !m || !v || step < 1) return CMRS_ERR_ARG;
  const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
  return launch_pdl(k_adam, (unsigned)grid_for(n, 256), 256, 0, as_stream(stream), n, params, grads, m, v, lr, beta1,
                    beta2, eps, c1, c2);
}

// ------------------------------------------------------------------ selection
// Padded forms the exhaustive sweep times must fit this many items; a form
// padded beyond it (more than twice the entries) is not a candidate.
static size_t pad_cap(int rows, int nnz) { return 2 * (size_t)nnz + 32 * ((size_t)rows / 16 + 2); }

static size_t select_ws(int rows, int cols, int nnz, int exhaustive) {
  size_t b = features_ws(rows) + align256(kNFeat * 8) + align256(64);
  if (exhaustive) {
    const size_t strips = (size_t)rows + 1;
    b += align256(strips * 4) + align256((size_t)std::max(nnz, 1) * 4) * 3 + align256((size_t)std::max(cols, 1) * 4) +
         align256((size_t)std::max(rows, 1) * 4);
    size_t s = 0;
    cmrs_from_csr_workspace(rows, nnz, 1, 0, CMRS_F32, &s);
    b += align256(s);
    // padded forms: StripPtr, items (packed + FP32 values) and the layout pass's workspace
    b += align256(((size_t)rows / 16 + 2) * 4) + 2 * align256(pad_cap(rows, nnz) * 4) + align256(256) +
         align256(((size_t)rows / 16 + 2) * 4) + align256(((size_t)rows / 16 + 2) * 8) + align256(((size_t)rows / 16 / 1024 + 2) * 8);
    b += align256(merge_workspace_bytes(nnz, CMRS_F32) + 4096);
  }
  return b;
}

// ------------------------------------------------------------------ training data
namespace cmrs {
namespace {
// Feature j's mean and population standard deviation over the B rows, summed
// in row order in FP64 (one thread per feature); scale = 1 / std, or 0 for a
// feature that does not vary (it then leaves the network's input).
__global__ void k_feat_stats(int B, int nin, const double *__restrict__ F, float *__restrict__ mean,
                             float *__restrict__ scale) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= nin) return;
  double s = 0.0;
  for (int n = 0; n < B; ++n) s = __dadd_rn(s, F[(size_t)n * nin + j]);
  const double m = __ddiv_rn(s, (double)B);
  double q = 0.0;
  for (int n = 0; n < B; ++n) {
    const double d = __dsub_rn(F[(size_t)n * nin + j], m);
    q = __dadd_rn(q, __dmul_rn(d, d));
  }
  const double sd = sqrt(__ddiv_rn(q, (double)B));
  mean[j] = (float)m;
  scale[j] = sd > 1e-12 ? (float)__ddiv_rn(1.0, sd) : 0.f;
}

// X = (F - mean) * scale in FP32, row-major [B][nin].
__global__ void k_feat_apply(int total, int nin, const double *__restrict__ F, const float *__restrict__ mean,
                             const float *__restrict__ scale, float *__restrict__ X) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= total) return;
  const int j = t % nin;
  X[t] = ((float)F[t] - mean[j]) * scale[j];
}

// T[n][c] = min(log2(t[n][c] / min_c t[n][c]), cap): each choice's cost
// relative to the row's best, one thread per row.
__global__ void k_cost_targets(int B, int nout, const double *__restrict__ times, float cap, float *__restrict__ T) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= B) return;
  const double *t = times + (size_t)n * nout;
  double best = t[0];
  for (int c = 1; c < nout; ++c) best = t[c] < best ? t[c] : best;
  for (int c = 0; c < nout; ++c) {
    const double r = log2(__ddiv_rn(t[c], best));
    T[(size_t)n * nout + c] = (float)(r < (double)cap ? r : (double)cap);
  }
}
}  // namespace
}  // namespace cmrs

extern "C" int cmrs_feature_norm(int B, int nin, const double *F, float *mean, float *scale, float *X, void *stream) {
  CMRS_TRACE();
  if (B < 1 || nin < 1 || !F || !mean || !scale) return CMRS_ERR_ARG;
  cudaStream_t st = as_stream(stream);
  k_feat_stats<<<(nin + 63) / 64, 64, 0, st>>>(B, nin, F, mean, scale);
  CMRS_LAUNCH_CHECK();
  if (X) {
    const long long total = (long long)B * nin;
    if (total >= (1LL << 31)) return CMRS_ERR_ARG;
    k_feat_apply<<<(int)ceil_div(total, 256), 256, 0, st>>>((int)total, nin, F, mean, scale, X);
    CMRS_LAUNCH_CHECK();
  }
  return CMRS_OK;
}

extern "C" int cmrs_feature_apply(int B, int nin, const double *F, const float *mean, const float *scale, float *X,
                                  void *stream) {
  CMRS_TRACE();
  const long long total = (long long)B * nin;
  if (B < 1 || nin < 1 || !F || !mean || !scale || !X || total >= (1LL << 31)) return CMRS_ERR_ARG;
  k_feat_apply<<<(int)ceil_div(total, 256), 256, 0, as_stream(stream)>>>((int)total, nin, F, mean, scale, X);
  CMRS_LAUNCH_CHECK();
  return CMRS_OK;
}

extern "C" int cmrs_cost_targets(int B, int nout, const double *times, float cap, float *T, void *stream) {
  CMRS_TRACE();
  if (B < 1 || nout < 1 || !times || !T || !(cap > 0.f)) return CMRS_ERR_ARG;
  k_cost_targets<<<(B + 127) / 128, 128, 0, as_stream(stream)>>>(B, nout, times, cap, T);
  CMRS_LAUNCH_CHECK();
  return CMRS_OK;
}

extern "C" int cmrs_select_strip_workspace(int rows, int cols, int nnz, int exhaustive, size_t *bytes) {
  if (rows < 1 || cols < 1 || nnz < 0 || !bytes) return CMRS_ERR_ARG;
  *bytes = select_ws(rows, cols, nnz, exhaustive);
  return CMRS_OK;
}

__global__ void k_fill(float *p, long long n, float v) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    p[i] = v;
}

extern "C" int cmrs_select_strip(int rows, int cols, int nnz, const int32_t *row_ptr, const int32_t *col_ind,
                                 const cmrs_selector *model, int *height_out, int *variant_out, int *slots_out,
                                 void *workspace, size_t workspace_bytes, void *stream) {
  CMRS_TRACE();
  if (rows < 1 || cols < 1 || nnz < 0 || !row_ptr || !height_out || !variant_out || !slots_out) return CMRS_ERR_ARG;
  const int exhaustive = model == nullptr;
  const size_t need = select_ws(rows, cols, nnz, exhaustive);
  if (!workspace || workspace_bytes < need || (reinterpret_cast<uintptr_t>(workspace) & 255)) return CMRS_ERR_WORKSPACE;
  cudaStream_t st = as_stream(stream);
  char *ws = reinterpret_cast<char *>(workspace);
  size_t off = features_ws(rows);
  double *feat = reinterpret_cast<double *>(ws + off);
  off += align256(kNFeat * 8);
  int *choice = reinterpret_cast<int *>(ws + off);
  off += align256(64);
  if (!exhaustive) {
    if (model->nin != kNFeat || model->nout != CMRS_SEL_CHOICES || model->nh < 1 || model->nh > 64 || !model->params ||
        !model->feat_mean || !model->feat_scale)
      return CMRS_ERR_ARG;
    int rc = cmrs_features(rows, nnz, row_ptr, col_ind, feat, workspace, features_ws(rows), stream);
    if (rc) return rc;
    const int nh = model->nh, nout = model->nout;  // nh <= 64: the network takes at most 34 KB of shared memory
    rc = launch_pdl(k_choose, 1, kMlpThreads, mlp_smem_floats(kNFeat, nh, nout) * 4, st, kNFeat, nh, nout, feat,
                    model->feat_mean, model->feat_scale, model->params, choice);
    if (rc) return rc;
    int c = 0;
    CMRS_CUDA_TRY(cudaMemcpyAsync(&c, choice, sizeof(int), cudaMemcpyDeviceToHost, st));
    CMRS_CUDA_TRY(cudaStreamSynchronize(st));
    if (c < 18) {
      *height_out = kHeights[c / 3];
      *variant_out = c % 3;
      *slots_out = 0;
    } else {
      *height_out = kPadChoice[c - 18][0];
      *variant_out = CMRS_VARIANT_PADDED;
      *slots_out = kPadChoice[c - 18][1];
    }
    return CMRS_OK;
  }
  // Exhaustive autotune (Section 6.2's brute force): convert with every
  // height and time every variant; the values are ones (timing does not
  // depend on them).
  int32_t *sp = reinterpret_cast<int32_t *>(ws + off);
  off += align256(((size_t)rows + 1) * 4);
  uint32_t *pk = reinterpret_cast<uint32_t *>(ws + off);
  off += align256((size_t)std::max(nnz, 1) * 4);
  float *val = reinterpret_cast<float *>(ws + off);
  off += align256((size_t)std::max(nnz, 1) * 4);
  float *ones = reinterpret_cast<float *>(ws + off);
  off += align256((size_t)std::max(nnz, 1) * 4);
  float *x = reinterpret_cast<float *>(ws + off);
  off += align256((size_t)cols * 4);
  float *y = reinterpret_cast<float *>(ws + off);
  off += align256((size_t)rows * 4);
  size_t cws = 0;
  cmrs_from_csr_workspace(rows, nnz, 1, 0, CMRS_F32, &cws);
  char *conv_ws = ws + off;
  off += align256(cws);
  const size_t cap = pad_cap(rows, nnz);
  int32_t *psp = reinterpret_cast<int32_t *>(ws + off);
  off += align256(((size_t)rows / 16 + 2) * 4);
  uint32_t *ppk = reinterpret_cast<uint32_t *>(ws + off);
  off += align256(cap * 4);
  float *pval = reinterpret_cast<float *>(ws + off);
  off += align256(cap * 4);
  char *pad_ws = ws + off;
  const size_t pad_ws_bytes = align256(256) + align256(((size_t)rows / 16 + 2) * 4) +
                              align256(((size_t)rows / 16 + 2) * 8) + align256(((size_t)rows / 16 / 1024 + 2) * 8);
  off += pad_ws_bytes;
  char *spmv_ws = ws + off;
  const size_t spmv_bytes = workspace_bytes - off;
  k_fill<<<grid_for(std::max(nnz, 1), 256), 256, 0, st>>>(ones, std::max(nnz, 1), 1.f);
  k_fill<<<grid_for(cols, 256), 256, 0, st>>>(x, cols, 1.f);
  CMRS_LAUNCH_CHECK();
  CMRS_CUDA_TRY(cudaMemsetAsync(spmv_ws, 0, 256, st));
  cudaEvent_t e0, e1;
  CMRS_CUDA_TRY(cudaEventCreate(&e0));
  CMRS_CUDA_TRY(cudaEventCreate(&e1));
  float best = 1e30f;
  int bh = 4, bv = 0, bm = 0, rc = CMRS_OK;
  auto time_one = [&](const cmrs_matrix *M, int v, int h, int m) {
    for (int w = 0; w < 2 && rc == CMRS_OK; ++w) rc = cmrs_spmv(M, x, y, v, spmv_ws, spmv_bytes, stream);
    cudaEventRecord(e0, st);
    for (int r = 0; r < 5 && rc == CMRS_OK; ++r) rc = cmrs_spmv(M, x, y, v, spmv_ws, spmv_bytes, stream);
    cudaEventRecord(e1, st);
    cudaError_t e = cudaEventSynchronize(e1);
    float ms = 0.f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
    if (e != cudaSuccess && rc == CMRS_OK) rc = set_cuda_error(e);
    if (rc == CMRS_OK && ms < best) {
      best = ms;
      bh = h;
      bv = v;
      bm = m;
    }
  };
  for (int hi = 0; hi < 6 && rc == CMRS_OK; ++hi) {
    cmrs_matrix A;
    rc = cmrs_from_csr(rows, cols, nnz, row_ptr, col_ind, ones, CMRS_F32, kHeights[hi], 0, CMRS_F32, sp, pk, val,
                       conv_ws, cws, stream, &A);
    for (int v = 0; v < 3 && rc == CMRS_OK; ++v) time_one(&A, v, kHeights[hi], 0);
    // the padded forms built from this height's CMRS
    for (int j = 0; j < 3 && rc == CMRS_OK; ++j) {
      if (kPadChoice[j][0] != kHeights[hi]) continue;
      int32_t npad = 0;
      rc = cmrs_pad_layout(&A, kPadChoice[j][1], psp, &npad, pad_ws, pad_ws_bytes, stream);
      if (rc == CMRS_OK && (size_t)npad <= cap) {
        cmrs_matrix P;
        rc = cmrs_pad_fill(&A, kPadChoice[j][1], psp, npad, ppk, pval, stream, &P);
        if (rc == CMRS_OK) time_one(&P, CMRS_VARIANT_PADDED, kHeights[hi], kPadChoice[j][1]);
      }
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc) return rc;
  *height_out = bh;
  *variant_out = bv;
  *slots_out = bm;
  return CMRS_OK;
}
