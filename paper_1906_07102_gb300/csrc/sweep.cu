// Single-plan gridding and degridding: the nearest / linear table kernels (the extended
// lookups are compiled in sweep_ext.cu), the spill pass, launch configuration.
#include <algorithm>

#include "sweep_body.cuh"

namespace lmg {
namespace {

// What gridding leaves to add after the sweep, a warp at a time: the spill rows of the items (none
// when the sweep added into a zeroed grid), and the merged chains of cut row pairs: one row of one pair
// is summed over the pair's chains, their rounding errors apart, and added to the grid once. One launch for both: a second one costs 3 us, a tenth of gridding 1000 visibilities.
__global__ void k_grid_spill(const Item* __restrict__ items, const int* __restrict__ counters, int item_cap, int W,
                            int RS, int N, const float2* __restrict__ spill, float2* __restrict__ grid, int merged,
                            const Cut* __restrict__ cuts, int part_cap, const float2* __restrict__ parts) {
  constexpr int S = strip_width(0);
  const int lane = threadIdx.x & 31, first = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int warps = (gridDim.x * blockDim.x) >> 5;
  if (spill != nullptr) {
    int nfront;
    const int total = work_total(counters, item_cap, nfront);
    for (int w = first; w < total; w += warps)
      spill_item<float>(items, nfront, item_cap, W, RS, N, S, spill, grid, w, lane, merged != 0);
  }
  const int total = min(counters[kCntCuts], part_cap) * (W + 1);
  for (int w = first; w < total; w += warps) {
    const Cut c = cuts[w / (W + 1)];
    const int row = w % (W + 1);
    const float2* p = parts + (static_cast<size_t>(c.part0) * (W + 1) + row) * (2 * S) + 2 * lane;
    unsigned long long s[2] = {0ull, 0ull}, e[2] = {0ull, 0ull};
    for (int k = 0; k < c.parts; ++k, p += (W + 1) * 2 * S) {
      const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p), r = *reinterpret_cast<const ulonglong2*>(p + S);
      two_sum_pair(s[0], e[0], v.x);
      two_sum_pair(s[1], e[1], v.y);
      e[0] = padd(e[0], r.x);
      e[1] = padd(e[1], r.y);
    }
    float2* dst = grid + static_cast<size_t>((c.r0 + row) % N) * N + c.strip * S + 2 * lane;
    red_add2(dst, f2unpack(padd(s[0], e[0])), f2unpack(padd(s[1], e[1])));
  }
}

void* kernel_for(int W, int dtype, int accum, bool degrid, bool ext, bool direct) {
  if (dtype) return sweep64_kernel(W, degrid, ext);
  return ext ? sweep_kernel_ext(W, accum, degrid, direct)
             : sweep_kernel_pick<false>(W, accum, degrid, direct);
}

}  // namespace

int ring_slots(int W) { return kD * ((W + kD - 1 + kD - 1) / kD); }

size_t sweep_smem_bytes(int W, int dtype, int Ms, bool table_in_smem, bool degrid, int warps) {
  if (dtype) return warps * sweep64_warp_bytes(W, degrid);
  const int Wp = table_stride(W, 0);
  const size_t tab = table_in_smem ? align16(size_t(Ms + 1) * Wp * sizeof(float)) : 0;
  return tab + size_t(warps) * stage_bytes(W, degrid);
}

int sweep_set_smem_limits(int W, int dtype, int accum, size_t smem_bytes, bool degrid, bool ext, bool direct) {
  void* k = kernel_for(W, dtype, accum, degrid, ext, direct);
  if (!k) return -1;
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem_bytes)) == cudaSuccess ? 0 : -1;
}

int sweep_occupancy(int W, int dtype, int accum, size_t smem_bytes, bool degrid, bool ext, bool direct, int warps,
                    int* blocks_per_sm) {
  void* k = kernel_for(W, dtype, accum, degrid, ext, direct);
  if (!k) return -1;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k, 32 * warps, smem_bytes) == cudaSuccess ? 0
                                                                                                                : -1;
}

int sweep_config(int W, int dtype, int Ms, bool degrid, size_t limit, bool* table_in_smem, int* warps) {
  if (dtype) {
    *table_in_smem = false;
    *warps = sweep64_warps();
    return 0;
  }
  const int Wp = table_stride(W, 0);
  *table_in_smem = align16(size_t(Ms + 1) * Wp * sizeof(float)) <= 96 * 1024;
  for (int pass = 0; pass < 2; ++pass) {
    for (int w = kWarps; w >= 1; w >>= 1) {
      if (sweep_smem_bytes(W, dtype, Ms, *table_in_smem, degrid, w) <= limit) {
        *warps = w;
        return 0;
      }
    }
    *table_in_smem = false;
  }
  return -1;
}

int grid_launch(const SweepArgs& a, cudaStream_t st) {
  void* k = kernel_for(a.W, a.dtype, a.accum, false, a.interp >= 2, a.direct != 0);
  if (!k) return -1;
  const size_t smem = sweep_smem_bytes(a.W, a.dtype, a.Ms, a.table_in_smem != 0, false, a.warps);
  cudaMemsetAsync(a.counters + kCntGridWork, 0, sizeof(int), st);
  if (a.direct) cudaMemsetAsync(a.grid, 0, size_t(a.N) * size_t(a.N) * (a.dtype ? 16 : 8), st);
  SweepArgs args = a;
  void* params[] = {&args};
  if (cudaLaunchKernel(k, dim3(a.grid_blocks), dim3(32 * a.warps), params, smem, st) != cudaSuccess) return -1;
  // complex64: a warp per item or cut row, 8 warps per CTA, at most 32 CTAs per SM (the rest in turn)
  const bool merged = merged_sums(a.W, a.accum != 0) && a.part_cap > 0;
  if (!a.direct || merged) {
    const int blocks = a.direct ? 2 * kSms : std::min((a.item_cap + 7) / 8, 32 * kSms);
    k_grid_spill<<<blocks, 256, 0, st>>>(a.items, a.counters, a.item_cap, a.W, ring_slots(a.W), a.N,
                                        a.direct ? nullptr : static_cast<const float2*>(a.spill),
                                        static_cast<float2*>(a.grid), merged_sums(a.W, a.accum != 0) ? 1 : 0, a.cuts,
                                         merged ? a.part_cap : 0, a.parts);
  }
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int degrid_launch(const SweepArgs& a, cudaStream_t st, bool zero_out) {
  void* k = kernel_for(a.W, a.dtype, 0, true, a.interp >= 2, false);
  if (!k) return -1;
  const size_t smem = sweep_smem_bytes(a.W, a.dtype, a.Ms, a.table_in_smem != 0, true, a.warps);
  // outputs start at zero: each record adds its partial sum (dropped positions stay zero)
  if (zero_out && a.nvis > 0) cudaMemsetAsync(a.vis_out, 0, size_t(a.nvis) * (a.dtype ? 16 : 8), st);
  cudaMemsetAsync(a.counters + kCntDegridWork, 0, sizeof(int), st);
  SweepArgs args = a;
  void* params[] = {&args};
  if (cudaLaunchKernel(k, dim3(a.grid_blocks), dim3(32 * a.warps), params, smem, st) != cudaSuccess) return -1;
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace lmg
