// Binning of visibility positions (support rule of Eq. 6) into strips of 64 (complex64) or
// 32 (complex128) columns sorted by pairs of support-start rows, and balanced work items for
// the sweep kernels.
//
// Pipeline (all on one stream, no host synchronisation):
//   1. k_bin_count   per visibility: float64 product to cells, exact fixed-point support
//                    rule, strip keys (one, or for complex64 two when the support crosses into
//                    the next strip); the bucket counter's returned value is the record's rank.
//   2. scan          exclusive prefix sum of the bucket counts (strip-major, row-minor).
//   3. k_bin_scatter positions recomputed from (u, v) (measured cheaper than storing a
//                    decoded 16-byte position per visibility and reloading it), records
//                    of each pair of rows (2m, 2m+1) of a strip -- the row group
//                    the sweeps stage together -- to the pair's range, dealt so that any 32
//                    consecutive records sample the whole pair (see dealt_position).
//   4. k_make_items  per strip and block of rows: items holding about item_target records,
//                    of whole row pairs (the sweeps' row groups) or parts of a dense pair.
// With a track layout (positions stored sample-major, k = t * tracks + b) passes 1 and 3
// follow each track instead (k_bin_count_tracks, k_bin_scatter_tracks).
#include <cuda_runtime.h>

#include "device_common.cuh"
#include "kernels.h"

namespace lmg {
namespace {

// i mod N in [0, N); positions inside the grid (the usual case) take no division.
__device__ __forceinline__ int wrap_index(long long i, int N) {
  if (static_cast<unsigned long long>(i) < static_cast<unsigned long long>(N)) return static_cast<int>(i);
  long long r = i % N;
  if (r < 0) r += N;
  return static_cast<int>(r);
}

// Support start (grid indices, wrapped to [0, N)) and table coordinates of position p =
// (u, v); false for a dropped position (product not finite or |u| N pixel_scale >= 2^30).
__device__ __forceinline__ bool vis_position(double2 p, double scale2, int W, int N, VisPos& vp,
                                             double2* delta = nullptr) {
  long long U, V;
  if (!fixed_position(p.x, scale2, U) || !fixed_position(p.y, scale2, V)) return false;
  if (delta) *delta = make_double2(quantisation_residual(p.x, scale2, U), quantisation_residual(p.y, scale2, V));
  long long n0, m0;
  support_start(U, W, n0, vp.su);
  support_start(V, W, m0, vp.sv);
  vp.x0 = wrap_index(n0 + N / 2, N);
  vp.y0 = wrap_index(m0 + N / 2, N);
  return true;
}

// Strip of a support-start column and the column inside it (strip_w is a power of two).
__device__ __forceinline__ int strip_of(int x0, int strip_w) { return x0 >> (__ffs(strip_w) - 1); }
__device__ __forceinline__ int col_in_strip(int x0, int strip_w) { return x0 & (strip_w - 1); }
__device__ __forceinline__ int next_strip(int strip, int n_strips) { return strip + 1 == n_strips ? 0 : strip + 1; }

// Pass 1: positions to grid cells (support rule), bucket keys, and each record's rank in
// its bucket (the value returned by the bucket counter), so that pass 2 needs no atomics.
// Each thread takes kCountIlp positions per iteration so that their bucket atomics are in
// flight together.
constexpr int kCountIlp = 4;

__global__ void k_bin_count(const double* __restrict__ uv, long long nvis, double scale2, int W, int Wx,
                            int N, int n_strips, int strip_w, int2* __restrict__ rank, int* __restrict__ hist,
                            int* __restrict__ counters, double2* __restrict__ frac) {
  const int lane = threadIdx.x & 31;  // for the dropped-position count
  const long long span = static_cast<long long>(blockDim.x) * kCountIlp;
  const long long stride = static_cast<long long>(gridDim.x) * span;
  for (long long base = static_cast<long long>(blockIdx.x) * span; base < nvis; base += stride) {
    VisPos vp[kCountIlp];
    int key1[kCountIlp], key2[kCountIlp];
    bool bad[kCountIlp];
#pragma unroll
    for (int u = 0; u < kCountIlp; ++u) {
      const long long k = base + u * blockDim.x + threadIdx.x;
      key1[u] = key2[u] = -1;
      bad[u] = false;
      vp[u] = VisPos{-1, 0, 0u, 0u};
      if (k < nvis) {
        double2 dl = make_double2(0.0, 0.0);
        const bool ok = vis_position(reinterpret_cast<const double2*>(uv)[k], scale2, W, N, vp[u],
                                     frac != nullptr ? &dl : nullptr);
        if (frac != nullptr) frac[k] = dl;
        if (ok) {
          const int strip = strip_of(vp[u].x0, strip_w);
          key1[u] = strip * N + vp[u].y0;
          if (col_in_strip(vp[u].x0, strip_w) + Wx > strip_w) key2[u] = next_strip(strip, n_strips) * N + vp[u].y0;
        } else {
          bad[u] = true;
        }
      }
    }
    int2 rk[kCountIlp];
#pragma unroll
    for (int u = 0; u < kCountIlp; ++u) {
      rk[u].x = key1[u] >= 0 ? atomicAdd(hist + key1[u], 1) : 0;
      rk[u].y = key2[u] >= 0 ? atomicAdd(hist + key2[u], 1) : 0;
    }
#pragma unroll
    for (int u = 0; u < kCountIlp; ++u) {
      const long long k = base + u * blockDim.x + threadIdx.x;
      if (k < nvis) rank[k] = rk[u];
      const unsigned nb = __popc(__ballot_sync(0xffffffffu, bad[u]));
      if (lane == 0 && nb) atomicAdd(counters + kCntBad, static_cast<int>(nb));
    }
  }
}

// Pass 1 where many positions share few buckets (a coarse grid): a CTA counts kDensePer positions a
// thread in shared memory and takes each bucket's ranks from the global counter at once. One
// counter update a record queues at the hot buckets' addresses: 4.1M visibilities on a 256^2
// grid (1024 buckets) took 524 us that way, 71 this way. From kDenseBuckets buckets on
// clearing and adding up the CTA's counters costs as much as it saves.
constexpr int kDenseThreads = 512;
constexpr int kDensePer = 8;
constexpr int kDenseBuckets = 4096;
constexpr int kDenseCount = 64;  // positions a bucket, on average

__global__ void __launch_bounds__(kDenseThreads)
    k_bin_count_dense(const double* __restrict__ uv, long long nvis, double scale2, int W, int Wx, int N, int n_strips,
                      int strip_w, int2* __restrict__ rank, int* __restrict__ hist, int* __restrict__ counters,
                      double2* __restrict__ frac) {
  __shared__ int s_hist[kDenseBuckets];
  const int L = n_strips * N, lane = threadIdx.x & 31;
  constexpr int kSpan = kDenseThreads * kDensePer;
  for (long long base = static_cast<long long>(blockIdx.x) * kSpan; base < nvis;
       base += static_cast<long long>(gridDim.x) * kSpan) {
    for (int i = threadIdx.x; i < L; i += kDenseThreads) s_hist[i] = 0;
    __syncthreads();
    int key1[kDensePer], key2[kDensePer];
    int2 rk[kDensePer];
#pragma unroll
    for (int u = 0; u < kDensePer; ++u) {
      const long long k = base + u * kDenseThreads + threadIdx.x;
      key1[u] = key2[u] = -1;
      rk[u] = make_int2(0, 0);
      bool bad = false;
      if (k < nvis) {
        VisPos vp{-1, 0, 0u, 0u};
        double2 dl = make_double2(0.0, 0.0);
        const bool ok = vis_position(reinterpret_cast<const double2*>(uv)[k], scale2, W, N, vp,
                                     frac != nullptr ? &dl : nullptr);
        if (frac != nullptr) frac[k] = dl;
        bad = !ok;
        if (ok) {
          const int strip = strip_of(vp.x0, strip_w);
          key1[u] = strip * N + vp.y0;
          if (col_in_strip(vp.x0, strip_w) + Wx > strip_w) key2[u] = next_strip(strip, n_strips) * N + vp.y0;
          rk[u].x = atomicAdd(s_hist + key1[u], 1);
          if (key2[u] >= 0) rk[u].y = atomicAdd(s_hist + key2[u], 1);
        }
      }
      const unsigned nb = __popc(__ballot_sync(0xffffffffu, bad));
      if (lane == 0 && nb) atomicAdd(counters + kCntBad, static_cast<int>(nb));
    }
    __syncthreads();
    for (int i = threadIdx.x; i < L; i += kDenseThreads) {
      const int n = s_hist[i];
      if (n > 0) s_hist[i] = atomicAdd(hist + i, n);
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kDensePer; ++u) {
      const long long k = base + u * kDenseThreads + threadIdx.x;
      if (key1[u] >= 0) rk[u].x += s_hist[key1[u]];
      if (key2[u] >= 0) rk[u].y += s_hist[key2[u]];
      if (k < nvis) rank[k] = rk[u];
    }
    __syncthreads();
  }
}

// Exclusive scan, stage 1: per-chunk sums.
constexpr int kScanThreads = 256;
constexpr int kScanPer = 16;
constexpr int kScanChunk = kScanThreads * kScanPer;

__global__ void k_scan_partials(const int* __restrict__ in, long long n, int* __restrict__ partial) {
  __shared__ int warp_sums[kScanThreads / 32];
  const long long base = static_cast<long long>(blockIdx.x) * kScanChunk + threadIdx.x * kScanPer;
  int s = 0;
#pragma unroll
  for (int i = 0; i < kScanPer; ++i)
    if (base + i < n) s += in[base + i];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) warp_sums[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
    for (int w = 0; w < kScanThreads / 32; ++w) t += warp_sums[w];
    partial[blockIdx.x] = t;
  }
}

// Stage 2: exclusive scan within each chunk plus the chunk's offset, the sum of the
// preceding chunks' totals (each CTA adds them up itself: a few thousand at most, cheaper
// than a separate launch); writes offsets[0..n].
__global__ void k_scan_final(const int* __restrict__ in, long long n, const int* __restrict__ partial,
                             int* __restrict__ offsets) {
  __shared__ int warp_sums[kScanThreads / 32];
  __shared__ int chunk_base;
  {
    int c = 0;
    for (int k = threadIdx.x; k < static_cast<int>(blockIdx.x); k += blockDim.x) c += partial[k];
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if ((threadIdx.x & 31) == 0) warp_sums[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
      int t = 0;
      for (int w = 0; w < kScanThreads / 32; ++w) t += warp_sums[w];
      chunk_base = t;
    }
    __syncthreads();
  }
  const long long base = static_cast<long long>(blockIdx.x) * kScanChunk + threadIdx.x * kScanPer;
  int v[kScanPer];
  int s = 0;
#pragma unroll
  for (int i = 0; i < kScanPer; ++i) {
    v[i] = (base + i < n) ? in[base + i] : 0;
    s += v[i];
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int x = s;
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_sums[w] = x;
  __syncthreads();
  int woff = 0;
  for (int k = 0; k < w; ++k) woff += warp_sums[k];
  int run = chunk_base + woff + x - s;
#pragma unroll
  for (int i = 0; i < kScanPer; ++i) {
    if (base + i < n) offsets[base + i] = run;
    run += v[i];
  }
  if (base + kScanPer >= n && base < n) offsets[n] = run;  // thread holding the last element
}

// The whole scan in one CTA, for up to kScanOne buckets (a grid of 1024^2 complex64): at that size
// each of the two launches above costs more than the work, so long as a thread's 16 buckets move as
// four 16-byte words (binning 20,000 visibilities, 512^2: 26.8 us, 32.9 with the two launches;
// 1024^2: 30.4 and 34.6, and 38 with single loads here).
constexpr int kScanOneThreads = 1024;
constexpr int kScanOne = kScanOneThreads * kScanPer;

__global__ void __launch_bounds__(kScanOneThreads)
    k_scan_one(const int* __restrict__ in, int n, int* __restrict__ offsets) {
  __shared__ int warp_sums[kScanOneThreads / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, base = threadIdx.x * kScanPer;
  // 16-byte loads and stores: n is a whole number of strips of N >= 64 rows, N a multiple of 32
  int v[kScanPer];
  int s = 0;
#pragma unroll
  for (int i = 0; i < kScanPer; i += 4) {
    const int4 q = base + i < n ? *reinterpret_cast<const int4*>(in + base + i) : make_int4(0, 0, 0, 0);
    v[i] = q.x;
    v[i + 1] = q.y;
    v[i + 2] = q.z;
    v[i + 3] = q.w;
    s += (q.x + q.y) + (q.z + q.w);
  }
  int x = s;
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_sums[w] = x;
  __syncthreads();
  int t = warp_sums[lane];
  const int own = t;
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, t, o);
    if (lane >= o) t += y;
  }
  int run = __shfl_sync(0xffffffffu, t - own, w) + x - s;
#pragma unroll
  for (int i = 0; i < kScanPer; i += 4) {
    const int4 q = make_int4(run, run + v[i], run + v[i] + v[i + 1], run + v[i] + v[i + 1] + v[i + 2]);
    if (base + i < n) *reinterpret_cast<int4*>(offsets + base + i) = q;
    run = q.w + v[i + 3];
  }
  if (threadIdx.x == kScanOneThreads - 1) offsets[n] = run;
}

// Pass 2: every record to offsets[bucket] + rank (no atomics).
// Position of the record of rank rho (0 .. n-1, in arrival order) inside its row pair of
// n records. Records of one baseline arrive in time order and land in nearby cells, so
// consecutive ranks cluster on a few columns; the sweeps give each lane the records that
// cover its column, so a chunk of clustered records leaves most lanes idle. The pair is
// dealt into nc = ceil(n / 32) runs, run j holding the ranks j, j + nc, j + 2 nc, ...
// (q or q + 1 of them, q = n / nc), so that any 32 consecutive positions hold ranks
// spread over the whole pair.
__device__ __forceinline__ int dealt_position(int rho, int n) {
  if (n <= 32) return rho;
  const int nc = (n + 31) >> 5, q = n / nc, r = n - q * nc;
  const int j = rho % nc;
  return j * q + min(j, r) + rho / nc;
}

__global__ void k_bin_scatter(const double* __restrict__ uv, double scale2, const int2* __restrict__ rank,
                              long long nvis, int W, int Wx, int N, int n_strips, int strip_w,
                              const int* __restrict__ offsets, Rec* __restrict__ recs) {
  // kCountIlp visibilities per thread per iteration: their position, rank and offset loads
  // are in flight together (the pass is bound by its random L2 requests and their latency).
  // (u, v) and the ranks are read for the last time here: streaming loads (evict first)
  // leave the L2 to the offsets and the records being written.
  const long long span = static_cast<long long>(blockDim.x) * kCountIlp;
  const long long stride = static_cast<long long>(gridDim.x) * span;
  for (long long base = static_cast<long long>(blockIdx.x) * span; base < nvis; base += stride) {
    VisPos vp[kCountIlp];
    int2 rk[kCountIlp];
#pragma unroll
    for (int u = 0; u < kCountIlp; ++u) {
      const long long k = base + u * blockDim.x + threadIdx.x;
      vp[u] = VisPos{-1, 0, 0u, 0u};
      rk[u] = make_int2(0, 0);
      if (k < nvis) {
        rk[u] = __ldcs(rank + k);
        vis_position(__ldcs(reinterpret_cast<const double2*>(uv) + k), scale2, W, N, vp[u]);
      }
    }
    int g1[kCountIlp], g2[kCountIlp];  // bucket pair bases (-1: none)
#pragma unroll
    for (int u = 0; u < kCountIlp; ++u) {
      g1[u] = g2[u] = -1;
      if (vp[u].x0 >= 0) {
        const int strip = strip_of(vp[u].x0, strip_w), xr = col_in_strip(vp[u].x0, strip_w);
        const int pair_row = vp[u].y0 & ~1;
        g1[u] = strip * N + pair_row;
        if (xr + Wx > strip_w) g2[u] = next_strip(strip, n_strips) * N + pair_row;
      }
    }
    // offsets of the pair's two rows and of the next pair (g is even: one 8-byte load and one
    // 4-byte load per record)
    int o1[kCountIlp][3], o2[kCountIlp][3];
#pragma unroll
    for (int u = 0; u < kCountIlp; ++u) {
      const int2 a1 = g1[u] >= 0 ? *reinterpret_cast<const int2*>(offsets + g1[u]) : make_int2(0, 0);
      const int2 a2 = g2[u] >= 0 ? *reinterpret_cast<const int2*>(offsets + g2[u]) : make_int2(0, 0);
      o1[u][0] = a1.x;
      o1[u][1] = a1.y;
      o1[u][2] = g1[u] >= 0 ? offsets[g1[u] + 2] : 0;
      o2[u][0] = a2.x;
      o2[u][1] = a2.y;
      o2[u][2] = g2[u] >= 0 ? offsets[g2[u] + 2] : 0;
    }
#pragma unroll
    for (int u = 0; u < kCountIlp; ++u) {
      if (g1[u] < 0) continue;
      const long long k = base + u * blockDim.x + threadIdx.x;
      const int odd = vp[u].y0 & 1, xr = col_in_strip(vp[u].x0, strip_w);
      // row pair (y0 & ~1, y0 | 1) of the strip: [offsets[g], offsets[g + 2])
      recs[o1[u][0] + dealt_position((odd ? o1[u][1] - o1[u][0] : 0) + rk[u].x, o1[u][2] - o1[u][0])] =
          Rec{static_cast<unsigned>(k), rec_pack(vp[u].y0, xr), vp[u].su, vp[u].sv};
      if (g2[u] >= 0)
        recs[o2[u][0] + dealt_position((odd ? o2[u][1] - o2[u][0] : 0) + rk[u].y, o2[u][2] - o2[u][0])] =
            Rec{static_cast<unsigned>(k), rec_pack(vp[u].y0, xr - strip_w), vp[u].su, vp[u].sv};
    }
  }
}

// Track-ordered binning. With the positions stored sample-major (k = t * tracks + b: one
// sample of every track, then the next sample), thread g follows track b = g mod tracks over
// kTrackChunk consecutive samples (chunk g / tracks); the lanes of a warp read neighbouring
// tracks at the same sample, so the position loads stay coalesced. Along a track the support
// moves by at most a few cells per sample and consecutive samples fall in the same bucket
// (strip, row) in runs (5.9 samples on average on 6 h Earth-rotation tracks with 64-column
// strips). The counting pass takes one bucket atomic per run and stores the rank it returns
// (the rank of the run's first record) at the run's first visibility; the placement pass walks
// the same runs and gives record j of a run the rank + j, loading that rank and the bucket's
// offsets once per run. Runs end where the bucket changes (a dropped position ends one) and at
// the end of a chunk, identically in both passes. Results do not depend on `tracks`: any value
// bins correctly; it only sets the order of the records within a bucket and the cost.
constexpr int kTrackChunk = 32;

__device__ __forceinline__ void bucket_keys(const VisPos& vp, int Wx, int N, int n_strips, int strip_w, int& key1,
                                            int& key2) {
  const int strip = strip_of(vp.x0, strip_w);
  key1 = strip * N + vp.y0;
  key2 = col_in_strip(vp.x0, strip_w) + Wx > strip_w ? next_strip(strip, n_strips) * N + vp.y0 : -1;
}

__global__ void k_bin_count_tracks(const double* __restrict__ uv, long long nvis, long long tracks, double scale2,
                                   int W, int Wx, int N, int n_strips, int strip_w, int2* __restrict__ rank,
                                   int* __restrict__ hist, int* __restrict__ counters, double2* __restrict__ frac) {
  const double2* uv2 = reinterpret_cast<const double2*>(uv);
  int* rank1 = reinterpret_cast<int*>(rank);  // rank[k].x = rank1[2 k], rank[k].y = rank1[2 k + 1]
  const long long n_t = (nvis + tracks - 1) / tracks;
  const long long n_threads = tracks * ((n_t + kTrackChunk - 1) / kTrackChunk);
  for (long long g = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; g < n_threads;
       g += static_cast<long long>(gridDim.x) * blockDim.x) {
    const long long b = g % tracks, t0 = (g / tracks) * kTrackChunk;
    const long long k_end = min(nvis, min(n_t, t0 + kTrackChunk) * tracks);
    int cur1 = -1, len1 = 0, cur2 = -1, len2 = 0;
    long long start1 = 0, start2 = 0;
    // the rank of a run is stored at the next flush, so that the atomic's round trip overlaps
    // the samples between (a store of its value right away would wait for it)
    long long pend1 = -1, pend2 = -1;
    int pval1 = 0, pval2 = 0;
    for (long long k = t0 * tracks + b; k < k_end; k += tracks) {
      VisPos vp{0, 0, 0u, 0u};
      double2 dl = make_double2(0.0, 0.0);
      const bool ok = vis_position(uv2[k], scale2, W, N, vp, frac != nullptr ? &dl : nullptr);
      if (frac != nullptr) frac[k] = dl;
      int key1 = -1, key2 = -1;
      if (ok) bucket_keys(vp, Wx, N, n_strips, strip_w, key1, key2);
      else atomicAdd(counters + kCntBad, 1);
      if (key1 != cur1) {
        if (len1 > 0) {
          if (pend1 >= 0) rank1[2 * pend1] = pval1;
          pval1 = atomicAdd(hist + cur1, len1);
          pend1 = start1;
        }
        cur1 = key1;
        start1 = k;
        len1 = 0;
      }
      len1 += key1 >= 0;
      if (key2 != cur2) {
        if (len2 > 0) {
          if (pend2 >= 0) rank1[2 * pend2 + 1] = pval2;
          pval2 = atomicAdd(hist + cur2, len2);
          pend2 = start2;
        }
        cur2 = key2;
        start2 = k;
        len2 = 0;
      }
      len2 += key2 >= 0;
    }
    if (len1 > 0) {
      if (pend1 >= 0) rank1[2 * pend1] = pval1;
      pval1 = atomicAdd(hist + cur1, len1);
      pend1 = start1;
    }
    if (len2 > 0) {
      if (pend2 >= 0) rank1[2 * pend2 + 1] = pval2;
      pval2 = atomicAdd(hist + cur2, len2);
      pend2 = start2;
    }
    if (pend1 >= 0) rank1[2 * pend1] = pval1;
    if (pend2 >= 0) rank1[2 * pend2 + 1] = pval2;
  }
}

// Placement of the records of one run: the pair's base and the dealt position (see
// dealt_position) of rank rho = row offset + run rank + j, kept as rho = i nc + jj so that
// each further record of the run costs no division.
struct RunPlace {
  int base, nc, q, r, jj, i;
  __device__ __forceinline__ void start(const int* __restrict__ offsets, int key, int rank0) {
    const int g = key & ~1;  // N is even: the pair's first row has an even key
    const int2 a = *reinterpret_cast<const int2*>(offsets + g);
    const int n = offsets[g + 2] - a.x;
    const int rho = ((key & 1) ? a.y - a.x : 0) + rank0;
    base = a.x;
    nc = max(1, (n + 31) >> 5);
    q = n / nc;
    r = n - q * nc;
    i = rho / nc;
    jj = rho - i * nc;
  }
  __device__ __forceinline__ int next() {
    const int pos = base + jj * q + min(jj, r) + i;
    if (++jj == nc) {
      jj = 0;
      ++i;
    }
    return pos;
  }
};

__global__ void k_bin_scatter_tracks(const double* __restrict__ uv, double scale2, const int2* __restrict__ rank,
                                     long long nvis, long long tracks, int W, int Wx, int N, int n_strips,
                                     int strip_w, const int* __restrict__ offsets, Rec* __restrict__ recs) {
  const double2* uv2 = reinterpret_cast<const double2*>(uv);
  const int* rank1 = reinterpret_cast<const int*>(rank);
  const long long n_t = (nvis + tracks - 1) / tracks;
  const long long n_threads = tracks * ((n_t + kTrackChunk - 1) / kTrackChunk);
  for (long long g = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; g < n_threads;
       g += static_cast<long long>(gridDim.x) * blockDim.x) {
    const long long b = g % tracks, t0 = (g / tracks) * kTrackChunk;
    const long long k_end = min(nvis, min(n_t, t0 + kTrackChunk) * tracks);
    int cur1 = -1, cur2 = -1;
    RunPlace run1{}, run2{};
    for (long long k = t0 * tracks + b; k < k_end; k += tracks) {
      VisPos vp;
      const bool ok = vis_position(__ldcs(uv2 + k), scale2, W, N, vp);
      int key1 = -1, key2 = -1;
      if (ok) bucket_keys(vp, Wx, N, n_strips, strip_w, key1, key2);
      if (key1 != cur1) {
        cur1 = key1;
        if (key1 >= 0) run1.start(offsets, key1, __ldcs(rank1 + 2 * k));
      }
      if (key2 != cur2) {
        cur2 = key2;
        if (key2 >= 0) run2.start(offsets, key2, __ldcs(rank1 + 2 * k + 1));
      }
      if (key1 < 0) continue;
      const int xr = col_in_strip(vp.x0, strip_w);
      recs[run1.next()] = Rec{static_cast<unsigned>(k), rec_pack(vp.y0, xr), vp.su, vp.sv};
      if (key2 >= 0) recs[run2.next()] = Rec{static_cast<unsigned>(k), rec_pack(vp.y0, xr - strip_w), vp.su, vp.sv};
    }
  }
}

// One CTA per (strip, block of rows). Thread i holds row pair i of the block. Pairs are joined
// with their neighbours into items of equal counts, about target records each. With a
// target below kDenseUnit (few visibilities) they are joined in units of the pairs that W - 1
// rows take, up to kDenseUnit records: items of whole units meet in a cell at most two at a time,
// so that their sums do not depend on which is added first. Elsewhere items are cut at any pair,
// and a pair with 2 part records or more is cut into parts of one to two times part, one item
// each: a warp sweeps an item alone, and one dense pair near the uv origin, 40 times the target,
// is otherwise a serial chain that the whole launch waits for (4.1M visibilities on a 256^2 grid:
// 512 such items kept a fifth of the resident warps busy, and degridding took 4.4 ms, 0.43 with
// the cut).
// fine (complex128): items are cut at any pair, and parts are as small as items: those sweeps end in tails of long items (see item_target_for), and their sums
// meet at the strips' edges in any order anyway.
// Items per block are at most 1 + joined / target and, for a cut pair of n >= 2 part records, at most
// n / part parts and one more boundary between joined pairs: 3 n / (2 part). With part >= 3/2 target
// (complex64) that is 1 + count / target in all; with part = target (complex128) half as much again,
// where item_bound allows two records a visibility and there is one.
// Items with more than target/2 records are placed from the front of the array and the others
// from the back, so that the sweeps (which take items front to back, then back to front)
// start the heavy ones first. skip_empty: items without records are left out (the gridding
// sweep then adds into a zeroed grid; otherwise they store their rows' zeros).
constexpr int kMaxRowsPerBlock = 512;
constexpr int kItemThreads = kMaxRowsPerBlock / 2;
constexpr int kManyBlocks = 4 * kSms;
constexpr int kDenseUnit = 512;
// Parts that plain float32 gridding sums in one chain. Its accuracy on dense cells follows the
// length of its chains; 4.1M visibilities on a 256^2 grid, W = 12, relative image error and time:
// uncut 4.9e-6 in 4.40 ms, 12 parts 1.8e-6 in 1.86, 8 parts 1.2e-6 in 1.23, 4 parts 6.3e-7 in
// 0.74, one 4.4e-7 in 0.40; compensated 2.5e-7 in 1.17 (9.9 uncut). Eight keep the plain sums as
// clearly apart from the compensated ones as tests/test_gpu_precision.py holds them (3 times).
constexpr int kChain = 8;

__device__ __forceinline__ void put_item(const Item& it, int target, Item* __restrict__ items,
                                         int* __restrict__ counters, int cap) {
  int slot;
  if (2 * it.nrec > target) slot = atomicAdd(counters + kCntItems, 1);
  else slot = cap - 1 - atomicAdd(counters + kCntItemsBack, 1);
  if (slot >= 0 && slot < cap) items[slot] = it;
  else atomicOr(counters + kCntStatus, kStatusItemOverflow);
}

// k-th of n blocks counted from the middle one outwards. Items are taken up in about the order
// in which their blocks place them, and the longest (chains of a dense pair's parts, 16,000 records
// and more) lie around the uv origin, in the grid's middle: placed first they do not end the
// sweep alone (gridding and degridding 49.5M visibilities 5602 -> 5316 us, 4.1M 545 -> 520).
__device__ __forceinline__ int centre_out(int k, int n) { return n / 2 + ((k & 1) ? -((k + 1) >> 1) : k >> 1); }

__global__ void __launch_bounds__(kItemThreads)
    k_make_items(const int* __restrict__ offsets, int N, int W, int rows_per_block, int target, int part, int skip_empty,
                 int fine, Item* __restrict__ items, int* __restrict__ counters, int cap, Cut* __restrict__ cuts, int part_cap,
                 int per_place) {
  __shared__ int s_off[kItemThreads + 1];  // offset of each pair's first record
  __shared__ int s_pre[kItemThreads];      // records of joined pairs before each pair
  __shared__ unsigned s_start[kItemThreads / 32 + 1], s_cut[kItemThreads / 32];
  __shared__ int s_warp[kItemThreads / 32];
  const int nblk = (N + rows_per_block - 1) / rows_per_block;
  const int n_strips = gridDim.x / nblk;
  const int s = centre_out(blockIdx.x % n_strips, n_strips), b = centre_out(blockIdx.x / n_strips, nblk);
  const int rb = b * rows_per_block, np = (min(N, rb + rows_per_block) - rb) / 2;
  const int i = threadIdx.x, lane = i & 31, warp = i >> 5, nw = blockDim.x >> 5;
  const int* off = offsets + static_cast<long long>(s) * N + rb;
  for (int k = i; k <= np; k += blockDim.x) s_off[k] = off[2 * k];
  __syncthreads();
  // unit of pair i: u pairs, the last unit of the block with the remainder
  const int u = target < kDenseUnit && !fine ? max(1, W >> 1) : 1, nu = max(1, np / u);
  auto unit_first = [&](int k) { return min(k / u, nu - 1) * u; };
  auto dense_unit = [&](int first) {
    const int end = first / u == nu - 1 ? np : first + u;
    return u == 1 || s_off[end] - s_off[first] > kDenseUnit;
  };
  const bool in = i < np;
  const int first = in ? unit_first(i) : 0;
  const bool dense = in && dense_unit(first);
  const int n = in ? s_off[i + 1] - s_off[i] : 0;
  const bool cut = dense && n >= 2 * part;
  const int nj = cut ? 0 : n;
  int x = nj;
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_warp[warp] = x;
  const unsigned cm = __ballot_sync(0xffffffffu, cut);
  if (lane == 0) s_cut[warp] = cm;
  __syncthreads();
  int base = 0, joined = 0;
  for (int k = 0; k < nw; ++k) {
    base += k < warp ? s_warp[k] : 0;
    joined += s_warp[k];
  }
  const int pre = base + x - nj;
  // joined pairs go to m items of equal counts, as far as the places to cut allow
  const int m_items = max(1, (joined + target - 1) / target);
  // (pairs after the last record belong to the last item: one of their own would pass the bound)
  auto item_of = [&](int r) {
    return joined ? min(m_items - 1, static_cast<int>(static_cast<long long>(r) * m_items / joined)) : 0;
  };
  s_pre[i] = pre;
  __syncthreads();
  // a joined item starts at the block's first pair, after a cut pair, and where the running
  // count passes into the next item's share
  bool start = in && (cut || i == 0);
  if (in && !start && (dense || i == first)) {
    const int f = unit_first(i - 1), p = dense_unit(f) ? i - 1 : f;
    start = ((s_cut[(i - 1) >> 5] >> ((i - 1) & 31)) & 1u) || item_of(pre) != item_of(s_pre[p]);
  }
  const unsigned sm = __ballot_sync(0xffffffffu, start);
  if (lane == 0) s_start[warp] = sm;
  __syncthreads();
  if (start && !cut) {
    int w = warp;
    unsigned m = lane == 31 ? 0u : s_start[w] & (0xffffffffu << (lane + 1));
    while (!m && ++w < nw) m = s_start[w];
    const int end = m ? 32 * w + __ffs(m) - 1 : np;
    const int cnt = s_off[end] - s_off[i];
    if (cnt > 0 || !skip_empty)
      put_item(Item{s, rb + 2 * i, 2 * (end - i), cnt, s_off[i], cnt, cnt, -1}, target, items, counters, cap);
  }
  // cut pairs, a warp each, their parts over its lanes (one after another over the CTA, with a
  // barrier before and after each pair's update of the parts' counter, the 4.1M visibilities of
  // a 256^2 grid took 39 to 58 us here, 16 now)
  int k0 = 0;
  for (int w = 0; w < nw; ++w) {
    for (unsigned m = s_cut[w]; m; m &= m - 1) {
      if (k0++ % nw != warp) continue;
      const int p = 32 * w + __ffs(m) - 1;
      const int o0 = s_off[p], cnt = s_off[p + 1] - o0, parts = cnt / part;
      // merged chains of per_place parts or more, a place each; a single one needs none
      const int merged = per_place > 0 ? parts / per_place : 0;
      int place = -1;
      if (merged > 1) {
        if (lane == 0) {
          const int q = atomicAdd(counters + kCntParts, merged);
          place = q + merged <= part_cap ? q : -1;
          if (place >= 0) cuts[atomicAdd(counters + kCntCuts, 1)] = Cut{s, rb + 2 * p, q, merged};
          else atomicOr(counters + kCntStatus, kStatusItemOverflow);
        }
        place = __shfl_sync(0xffffffffu, place, 0);
      }
      // shares of a whole, the first of them one larger: where the k-th begins
      const int rec = cnt / parts, rec1 = cnt % parts;
      const int per = merged > 1 ? parts / merged : 1, per1 = merged > 1 ? parts % merged : 0;
      auto record = [&](int k) { return rec * k + min(k, rec1); };
      auto first_part = [&](int g) { return per * g + min(g, per1); };
      for (int k = lane; k < parts; k += 32) {
        const int a = record(k), e = record(k + 1);
        const int chain = fine ? e - a : (k % kChain == 0 ? record(min(k + kChain, parts)) - a : 0);
        int comp = k == 0 ? cnt : 0, part = -1;
        if (place >= 0) {
          const int larger = per1 * (per + 1);
          const int g = k < larger ? k / (per + 1) : per1 + (k - larger) / per;
          comp = k == first_part(g) ? record(first_part(g + 1)) - a : 0;
          part = place + g;
        }
        put_item(Item{s, rb + 2 * p, k == 0 ? 2 : 0, e - a, o0 + a, chain, comp, part}, target, items, counters, cap);
      }
    }
  }
}

}  // namespace

int bin_launch(const BinArgs& a, cudaStream_t st) {
  const long long L = static_cast<long long>(a.n_strips) * a.N;
  // the counters lie behind the bucket counts: one launch clears both
  if (a.counters != a.hist + L) return -1;
  cudaMemsetAsync(a.hist, 0, sizeof(int) * (L + kNumCounters), st);
  const int wx = a.one_record ? 1 : a.W;  // columns by which a support crosses into the next strip
  const int threads = 256;
  const long long want_c = (a.nvis + threads * kCountIlp - 1) / (threads * kCountIlp);
  const int blocks_c = static_cast<int>(want_c < a.max_blocks ? (want_c > 0 ? want_c : 1) : a.max_blocks);
  long long n_tthreads = 0;
  if (a.tracks > 0) {
    const long long n_t = (a.nvis + a.tracks - 1) / a.tracks;
    n_tthreads = a.tracks * ((n_t + kTrackChunk - 1) / kTrackChunk);
  }
  const long long want_t = (n_tthreads + threads - 1) / threads;
  const int blocks_t = static_cast<int>(want_t < a.max_blocks ? (want_t > 0 ? want_t : 1) : a.max_blocks);
  if (a.tracks > 0)
    k_bin_count_tracks<<<blocks_t, threads, 0, st>>>(a.uv, a.nvis, a.tracks, a.scale2, a.W, wx, a.N, a.n_strips,
                                                     a.strip, a.rank, a.hist, a.counters, a.frac);
  else if (L <= kDenseBuckets && a.nvis >= kDenseCount * L) {
    const long long want = (a.nvis + kDenseThreads * kDensePer - 1) / (kDenseThreads * kDensePer);
    k_bin_count_dense<<<static_cast<int>(want < a.max_blocks ? want : a.max_blocks), kDenseThreads, 0, st>>>(
        a.uv, a.nvis, a.scale2, a.W, wx, a.N, a.n_strips, a.strip, a.rank, a.hist, a.counters, a.frac);
  } else
    k_bin_count<<<blocks_c, threads, 0, st>>>(a.uv, a.nvis, a.scale2, a.W, wx, a.N, a.n_strips, a.strip, a.rank,
                                            a.hist, a.counters, a.frac);
  const int nchunks = static_cast<int>((L + kScanChunk - 1) / kScanChunk);
  if (L <= kScanOne) {
    k_scan_one<<<1, kScanOneThreads, 0, st>>>(a.hist, static_cast<int>(L), a.offsets);
  } else {
    k_scan_partials<<<nchunks, kScanThreads, 0, st>>>(a.hist, L, a.partial);
    k_scan_final<<<nchunks, kScanThreads, 0, st>>>(a.hist, L, a.partial, a.offsets);
  }
  if (a.tracks > 0)
    k_bin_scatter_tracks<<<blocks_t, threads, 0, st>>>(a.uv, a.scale2, a.rank, a.nvis, a.tracks, a.W, wx, a.N,
                                                       a.n_strips, a.strip, a.offsets, a.recs);
  else
    k_bin_scatter<<<blocks_c, threads, 0, st>>>(a.uv, a.scale2, a.rank, a.nvis, a.W, wx, a.N, a.n_strips, a.strip,
                                              a.offsets, a.recs);
  const int nblk = (a.N + a.rows_per_block - 1) / a.rows_per_block;
  const int ntask = a.n_strips * nblk;
  if (a.rows_per_block > kMaxRowsPerBlock) return -1;
  // Threads: at least the block's row pairs. On sparse grids with more than kManyBlocks blocks, those of
  // up to 64 rows take one warp each: wide CTAs and their barriers are then what the launch costs
  // (binning of 200,000 visibilities: complex128 16384^2, 131,072 blocks, 304 -> 170 us; complex64
  // 2560^2, 1600 blocks, 40 -> 38). With fewer blocks four warps share the cut pairs of the dense ones
  // (0.7M on 256^2, 16 blocks: 66 us, in one warp each 102); with dense blocks narrow CTAs, all
  // resident at once, would place the items in no order (4.1M on 4096^2, gridding and degridding
  // 529 to 598 us in place of 473 to 534).
  const bool narrow = a.rows_per_block <= 64 && ntask > kManyBlocks && a.nvis < 256ll * ntask;
  const int item_threads = narrow ? 32 : (a.rows_per_block <= 256 ? 128 : kItemThreads);
  const int per_place = a.part_cap > 0 ? (part_bound(a.nvis) + a.part_cap - 1) / a.part_cap : 0;
  k_make_items<<<ntask, item_threads, 0, st>>>(a.offsets, a.N, a.W, a.rows_per_block, a.item_target, a.part_target,
                                               a.skip_empty, a.one_record, a.items, a.counters, a.item_cap, a.cuts,
                                               a.part_cap, per_place);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// Records per work item. A warp sweeps an item alone, so a call with few visibilities wants
// small items: with 512 records each, the 20,000 visibilities of a 256^2 grid made 40 items for
// 2432 resident warps and the sweep took 50 us, as long as one item does. 32 items per SM give
// each warp about two; from 32 records down an item is all start-up (its grid rows and
// offsets); above 512 nothing is gained (best of {256 .. 2048} on 4.1M-visibility tracks).
// Between 256 and 512 the second item of some warps becomes a third, and whole 512s are faster: 2.0M
// visibilities, W = 8, 2048^2, gridding and degridding 123 + 122 us with 411 records, 109 + 108.
// Supports from kWideSupport on keep half as many warps and read or add W - 1 rows more than an
// item owns, so that cutting blocks of rows costs more than it balances once there is one for each warp:
// degridding 200,000 visibilities, W = 12, 4096^2: 149 us with 41 records, 122 with 512; 2.0M: 310 and
// 260. With fewer blocks it gains (W = 12, 2048^2: 59 us uncut, 50).
// complex128: 96 items per SM, of which 10 to 32 are swept at a time. A record costs its SM 325
// cycles at W = 14, an item's rows little beside it: with 32 items per SM, two to three a warp, the
// float64 pipe stood still for a sixth of the sweep. Gridding and degridding in us: 1.03M visibilities,
// W = 14 cubic, 2048^2: 1646 + 1666 -> 1311 + 1320; 0.40M, W = 9, 256^2: 644 + 653 -> 275 + 277.
static int per_item(long long nvis, int per_sm) {
  const long long t = nvis / (per_sm * kSms);
  return static_cast<int>(t < 32 ? 32 : (t > kMaxItem ? kMaxItem : t));
}

int item_target_for(long long nvis, int dtype, int W, long long blocks) {
  if (dtype) return per_item(nvis, 96);
  const int t = per_item(nvis, 32);
  if (W >= kWideSupport) return blocks >= kWideWarps ? kMaxItem : t;
  return t > kMaxItem / 2 ? kMaxItem : t;
}

int part_target_for(long long nvis, int dtype, int target) {
  if (dtype) return target;
  const int t = 4 * per_item(nvis, 32), least = (3 * target + 1) / 2;
  return t > least ? t : least;
}

// Work items that nvis positions (two records each at most) can make (see k_make_items).
long long item_bound(long long nvis, int n_strips, int N, int rows_per_block, int target) {
  const long long nblk = (N + rows_per_block - 1) / rows_per_block;
  return n_strips * nblk + 2 * nvis / target + 2;
}

// Complex64: a cut pair's n records give at most n / (4 target) parts, and nvis positions two records
// each; nvis / item_target_for(nvis, 0) is largest at max_vis or where the target passes 33.
int part_bound(long long max_vis) {
  const long long n = max_vis / 32 <= 32 * kSms ? max_vis / 32 : 33 * kSms;
  return static_cast<int>((n > max_vis / 512 ? n : max_vis / 512) / 2 + 1);
}

int item_target_within(long long nvis, int dtype, int W, int n_strips, int N, int rows_per_block, int cap) {
  const long long blocks = item_bound(0, n_strips, N, rows_per_block, 1) - 2, room = cap - blocks - 2;
  const long long least = room > 0 ? (2 * nvis + room - 1) / room : 0;
  const int t = item_target_for(nvis, dtype, W, blocks);
  return least > t ? static_cast<int>(least) : t;
}

int bin_scan_chunks(long long L) { return static_cast<int>((L + kScanChunk - 1) / kScanChunk); }

}  // namespace lmg
