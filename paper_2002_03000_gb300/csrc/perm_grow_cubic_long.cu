// perm_grow_cubic_long.cu -- the growth kernel's instances for the cubic lattice, longer walks (64-bit site keys).
#include "perm_grow.cuh"

namespace perm {

cudaError_t launch_cubic_long(const RunDev &P, int thresh_mode, int ctas, cudaStream_t stream) {
    return launch_form<3, unsigned long long>(P, thresh_mode, ctas, stream);
}
cudaError_t allow_cubic_long() { return allow_smem_all<3, unsigned long long>(); }

}  // namespace perm
