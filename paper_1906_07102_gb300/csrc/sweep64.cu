// Sweep kernels of complex128 plans, nearest / linear table lookups (sweep64_ext.cu: the extended
// lookups).
#include "sweep64_body.cuh"

namespace lmg {
namespace {

template <int W> size_t warp_bytes(bool degrid) { return degrid ? Lay64<W>::degrid_bytes : Lay64<W>::grid_bytes; }

}  // namespace

void* sweep64_kernel_ext(int W, bool degrid);
void* sweep64_kernel(int W, bool degrid, bool ext) {
  return ext ? sweep64_kernel_ext(W, degrid) : sweep64_pick<false>(W, degrid);
}

int sweep64_warps() { return kWarps64; }

size_t sweep64_warp_bytes(int W, bool degrid) {
  switch (W) {
    case 1: return warp_bytes<1>(degrid);
    case 2: return warp_bytes<2>(degrid);
    case 3: return warp_bytes<3>(degrid);
    case 4: return warp_bytes<4>(degrid);
    case 5: return warp_bytes<5>(degrid);
    case 6: return warp_bytes<6>(degrid);
    case 7: return warp_bytes<7>(degrid);
    case 8: return warp_bytes<8>(degrid);
    case 9: return warp_bytes<9>(degrid);
    case 10: return warp_bytes<10>(degrid);
    case 11: return warp_bytes<11>(degrid);
    case 12: return warp_bytes<12>(degrid);
    case 13: return warp_bytes<13>(degrid);
    case 14: return warp_bytes<14>(degrid);
    case 15: return warp_bytes<15>(degrid);
    case 16: return warp_bytes<16>(degrid);
    default: return 0;
  }
}

}  // namespace lmg
