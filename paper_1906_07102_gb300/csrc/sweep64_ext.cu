// Sweep kernels of complex128 plans, extended lookups (Lagrange of degree 2 and 3, direct
// calculation): see sweep64.cu.
#include "sweep64_body.cuh"

namespace lmg {

void* sweep64_kernel_ext(int W, bool degrid) { return sweep64_pick<true>(W, degrid); }

}  // namespace lmg
