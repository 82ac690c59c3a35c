// Launch interfaces of the device kernels (host-callable, defined in the .cu files).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace lmg {

// Nodes k = 0..Ng of the direct calculation's folded sums (Ng = 32, Appendix A).
constexpr int kDirectNodes = 33;

// Strip width of the binning and the sweeps: 64 columns for complex64 (two a lane), 32 for
// complex128 (rows in shared memory). dtype 0 = complex64, 1 = complex128.
__host__ __device__ constexpr int strip_width(int dtype) { return dtype ? 32 : 64; }

// Row stride (reals) of a device table: rows start on 16-byte boundaries and take an odd
// number of 16-byte units, so that 16-byte loads of random rows spread over the banks;
// entries W .. stride - 1 are zero.
__host__ __device__ constexpr int table_stride(int W, int dtype) {
  return ((((W * (dtype ? 8 : 4) + 15) / 16) | 1) * 16) / (dtype ? 8 : 4);
}

struct Rec;
struct Item;
struct Cut;

constexpr int kSms = 152;  // GB300

// counters[] slots (device ints, reset by bin_launch)
enum {
  kCntBad = 0,         // dropped positions
  kCntItems = 1,       // items placed from the front (heavy)
  kCntStatus = 2,      // device status word: kStatus* bits set by the kernels' own checks
  kCntItemsBack = 3,   // items placed from the back (light)
  kCntGridWork = 4,    // work counter of the gridding sweep
  kCntDegridWork = 5,  // work counter of the degridding sweep
  kCntCuts = 6,        // cut row pairs
  kCntParts = 7,       // their parts
  kNumCounters = 8
};

// Device status bits (counters[kCntStatus]); the host reports them as LMG_EDEVICE.
enum {
  kStatusItemOverflow = 1,  // more work items than the plan's capacity: the excess was dropped
};

struct BinArgs {
  const double* uv;
  long long nvis;
  double scale2;  // N * pixel_scale * 2^32
  int W, N, n_strips, strip;  // strip: columns per strip (strip_width)
  int one_record;  // a support that crosses into the next strip still makes one record (its strip's)
  int rows_per_block, item_target, part_target, item_cap;
  int skip_empty;  // leave out work items without records (gridding into a zeroed grid)
  int max_blocks;
  int* hist;       // n_strips * N, followed by the counters
  int* offsets;    // n_strips * N + 1
  int2* rank;      // max_vis: rank of the record(s) in their buckets (gridding reuses the memory: SweepArgs::parts)
  int* partial;    // scan chunk sums
  Rec* recs;       // 2 * max_vis
  Item* items;     // item_cap
  Cut* cuts;       // part_cap or NULL (no merged chains): the cut row pairs
  int part_cap;
  int* counters;   // kNumCounters, at hist + n_strips * N
  double2* frac;   // max_vis or NULL: per visibility (u_q - u, v_q - v) in cells, the residual
                   // of the 2^-32 quantisation (float64 plans: exact table fractions)
  long long tracks;  // > 0: positions ordered k = t * tracks + b (sample t of track b); the
                     // counting and placement passes then follow each track in runs of
                     // samples that share a bucket. 0: no order assumed.
};

// Fused kept-field transforms (fft.cu): complex64 plans with N = kXformN only.
constexpr int kXformN = 4096;
bool xform_supported(int dtype, long long N, long long n);
size_t xform_scratch_bytes(long long n);
int xform_set_limits();
int xform_image_launch(const void* grid, void* image, void* scratch, const float* h, const void* tw, int n,
                       cudaStream_t st);
int xform_model_launch(const void* image, void* grid, void* scratch, const float* h, const void* tw, int n,
                       cudaStream_t st);

int bin_launch(const BinArgs& a, cudaStream_t st);
int bin_scan_chunks(long long L);
constexpr int kMaxItem = 512;          // records
constexpr int kWideSupport = 9;        // from here on the float32 sweeps keep 8 warps per SM, 16 below
constexpr int kWideWarps = 8 * kSms;   // resident in all
int item_target_for(long long nvis, int dtype, int W, long long blocks);
// Records of one part of a cut row pair, about: at least 3/2 target (item_bound).
int part_target_for(long long nvis, int dtype, int target);
long long item_bound(long long nvis, int n_strips, int N, int rows_per_block, int target);
// Parts of cut row pairs that up to max_vis positions can make.
int part_bound(long long max_vis);
// item_target_for, raised until item_bound stays within cap items.
int item_target_within(long long nvis, int dtype, int W, int n_strips, int N, int rows_per_block, int cap);
// Gridding by adding into a zeroed grid instead of storing whole rows and adding spill rows, complex64
// (complex128 always adds): where the grid stays in L2 (129 MB, half of it at most), zeroing and vector
// reductions cost no DRAM traffic, and small items need no spill buffer and no pass over it.
constexpr bool grid_direct(long long N) { return N * N * 8 <= (48ll << 20); }
// Few visibilities for the grid: storing its rows, mostly zeros, as the sweep passes them is then cheaper
// than zeroing all and adding some. Gridding in us, stored and added: 20,000 on 2496^2 (W = 5) 31 and
// 38, on 2048^2 33 and 35, on 1600^2 36 and 30; 1000 on 1024^2 (W = 16) 31 and 38.
constexpr bool grid_sparse(long long N, long long nvis) { return nvis << 18 < N * N * N; }

struct SweepArgs {
  const Rec* recs;
  const int* offsets;
  const Item* items;
  int* counters;
  const void* table;  // device, (Ms+1) x Wp of the plan's real type
  int Wp, Ms, interp;
  int N, n_strips, strip;
  int W;
  int dtype;          // 0 float, 1 double
  int accum;          // 0 plain, 1 compensated (float only)
  int item_cap;
  int direct;         // gridding adds into a zeroed grid; else rows are stored once
  int grid_blocks;    // persistent CTAs
  int warps;          // warps per CTA (1..8)
  int table_in_smem;
  // gridding
  const void* vis;
  const void* weights;
  void* grid;
  void* spill;        // item_cap * ring rows * strip complex (not used when direct)
  int part_cap;       // merged chains there can be, 0 for none
  const Cut* cuts;    // their row pairs and their sums, [place][W + 1 rows][sum, rounding error][strip]
  float2* parts;
  // degridding
  const void* grid_in;
  void* vis_out;
  long long nvis;
  const double2* frac;  // float64 plans: quantisation residuals (BinArgs::frac), else NULL
};

int grid_launch(const SweepArgs& a, cudaStream_t st);
// Rows held in the sweep's rolling ring for support W (spill buffer rows per item).
int ring_slots(int W);
// zero_out: zero the outputs first (else the predictions are added to what is there)
int degrid_launch(const SweepArgs& a, cudaStream_t st, bool zero_out = true);
// Shared memory a sweep CTA needs (bytes) and CTAs per SM that fit; used to size launches.
size_t sweep_smem_bytes(int W, int dtype, int Ms, bool table_in_smem, bool degrid, int warps);
// ext: the kernels of the extended lookups (interp >= 2: Lagrange, direct calculation).
int sweep_set_smem_limits(int W, int dtype, int accum, size_t smem_bytes, bool degrid, bool ext, bool direct);
int sweep_occupancy(int W, int dtype, int accum, size_t smem_bytes, bool degrid, bool ext, bool direct, int warps,
                    int* blocks_per_sm);
// Kernel of the extended lookups (sweep_ext.cu).
void* sweep_kernel_ext(int W, int accum, bool degrid, bool direct);
// Kernels of complex128 plans (sweep64.cu), their warps per CTA and a warp's shared memory.
void* sweep64_kernel(int W, bool degrid, bool ext);
int sweep64_warps();
size_t sweep64_warp_bytes(int W, bool degrid);
// Warps per CTA and table placement so that a CTA's shared memory stays within `limit`.
int sweep_config(int W, int dtype, int Ms, bool degrid, size_t limit, bool* table_in_smem, int* warps);

// Grid correction (Eqs. 4, 15) and its adjoint.
int crop_correct_launch(const void* F, void* img, const void* h, int n_img, int N, int dtype, cudaStream_t st);
int pad_correct_launch(const void* img, void* P, const void* h, int n_img, int N, int dtype, cudaStream_t st);
// Pad + correct writing only the kept rows of P (the rest must already be zero).
int pad_rows_launch(const void* img, void* P, const void* h, int n_img, int N, int dtype, cudaStream_t st);

}  // namespace lmg
