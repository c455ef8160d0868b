// Instantiation of the FP32 shell-force kernel for pair diameters up to 4.
#include "lbe_shell_march.cuh"

namespace lbe {
cudaError_t launch_shell_march_4(const ShellMarchMaps &maps, ShellMarchArgs &A, cudaStream_t st) {
    return launch_shell_march_t<4>(maps, A, st);
}
}  // namespace lbe
