// perm_grow_cubic.cu -- the growth kernel's instances for the cubic lattice, n_max <= 512 (32-bit site keys).
#include "perm_grow.cuh"

namespace perm {

cudaError_t launch_cubic(const RunDev &P, int thresh_mode, int ctas, cudaStream_t stream) {
    return launch_form<3, uint32_t>(P, thresh_mode, ctas, stream);
}
cudaError_t allow_cubic() { return allow_smem_all<3, uint32_t>(); }

}  // namespace perm
