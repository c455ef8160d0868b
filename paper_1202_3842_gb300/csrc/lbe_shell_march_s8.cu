// Instantiation of the FP32 shell-force kernel for pair diameters up to 8.
#include "lbe_shell_march.cuh"

namespace lbe {
cudaError_t launch_shell_march_8(const ShellMarchMaps &maps, ShellMarchArgs &A, cudaStream_t st) {
    return launch_shell_march_t<8>(maps, A, st);
}
}  // namespace lbe
