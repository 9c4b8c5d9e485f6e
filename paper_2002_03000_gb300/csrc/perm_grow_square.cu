// perm_grow_square.cu -- the growth kernel's instances for the square lattice.
#include "perm_grow.cuh"

namespace perm {

cudaError_t launch_square(const RunDev &P, int thresh_mode, int ctas, cudaStream_t stream) {
    return launch_form<2, uint32_t>(P, thresh_mode, ctas, stream);
}
cudaError_t allow_square() { return allow_smem_all<2, uint32_t>(); }

}  // namespace perm
