// Instantiation of the FP64 shell-force kernel for pair diameters up to 4.
#include "lbe_shell_fixed.cuh"

namespace lbe {
cudaError_t launch_shell_fixed_4(const ShellMarchMaps &maps, FixedArgs &A, cudaStream_t st) {
    return launch_shell_fixed_t<4>(maps, A, st);
}
}  // namespace lbe
