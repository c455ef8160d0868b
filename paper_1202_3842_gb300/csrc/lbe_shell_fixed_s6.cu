// Instantiation of the FP64 shell-force kernel for pair diameters up to 6.
#include "lbe_shell_fixed.cuh"

namespace lbe {
cudaError_t launch_shell_fixed_6(const ShellMarchMaps &maps, FixedArgs &A, cudaStream_t st) {
    return launch_shell_fixed_t<6>(maps, A, st);
}
}  // namespace lbe
