// Dispatch of the shell-force kernels by precision and pair diameter, and the host-side shell helpers.
// FP32: every pair in one launch of the marching kernel (lbe_shell_march.cuh), instantiated for the largest
// pair diameter 4, 6 or 8 (the registers of a thread grow with it: 128, 166, 222, so four, three and two
// blocks of 128 threads per SM).  FP64: one launch per pair of the plain kernel (lbe_shell_kernels.cuh).
#include "lbe_device.cuh"
#include "lbe_launch.h"
#include "lbe_shell.cuh"
#include "lbe_shell_march.cuh"

namespace lbe {

template <typename T, int S>
cudaError_t launch_one(const ShellLaunch &L, cudaStream_t st);
cudaError_t launch_shell_march_4(const ShellMarchMaps &maps, ShellMarchArgs &A, cudaStream_t st);
cudaError_t launch_shell_march_6(const ShellMarchMaps &maps, ShellMarchArgs &A, cudaStream_t st);
cudaError_t launch_shell_march_8(const ShellMarchMaps &maps, ShellMarchArgs &A, cudaStream_t st);

cudaError_t launch_shell_march(int Smax, const ShellMarchMaps &maps, ShellMarchArgs &A, cudaStream_t st) {
    if (Smax < 1 || Smax > 8) return cudaErrorInvalidValue;
    return Smax <= 4 ? launch_shell_march_4(maps, A, st)
                     : (Smax <= 6 ? launch_shell_march_6(maps, A, st) : launch_shell_march_8(maps, A, st));
}

__global__ void k_fill(float *__restrict__ p, long long n, float v) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        p[i] = v;
}
cudaError_t launch_fill(float *p, long long n, float v, cudaStream_t st) {
    const long long nb = (n + 255) / 256;
    k_fill<<<(unsigned)(nb < 8 * 152 ? nb : 8 * 152), 256, 0, st>>>(p, n, v);
    return cudaGetLastError();
}

cudaError_t launch_shell_force(int S, const ShellLaunch &L, cudaStream_t st) {
    switch (S) {
        case 1: return launch_one<double, 1>(L, st);
        case 2: return launch_one<double, 2>(L, st);
        case 3: return launch_one<double, 3>(L, st);
        case 4: return launch_one<double, 4>(L, st);
        case 5: return launch_one<double, 5>(L, st);
        case 6: return launch_one<double, 6>(L, st);
        case 7: return launch_one<double, 7>(L, st);
        default: return cudaErrorInvalidValue;
    }
}

bool shell_supported(bool fp64, int S) { return S >= 1 && S <= (fp64 ? 7 : 8); }

// Box of the shell-transpose tiles (lbe_adj_shell.cuh, dispatched in lbe_adjoint.cu).  FP32: the
// interleaved 8-byte (Lambda, g Lambda) elements of a 32 x 16 tile (32 x 8 at S = 8), the tile the
// transpose itself runs; FP64: the forward kernel's box of two separate planes.
void adj_shell_box(bool fp64, int S, int *bx, int *by) {
    if (!fp64) {
        *bx = ((32 + 2 * S + 1) + 1) / 2 * 2;
        *by = (S <= 7 ? 16 : 8) + 2 * S;
        return;
    }
    shell_box(true, S, bx, by);
}

void shell_box(bool fp64, int S, int *bx, int *by) {
    if (!fp64) {  // ShellMarchTile
        *bx = 32 + 2 * ((S + 3) / 4 * 4);
        *by = SM_TY + 2 * S;
        return;
    }
#define LBE_BOX(s)                              \
    case s:                                     \
        *bx = ShellTile<double, s>::BX;         \
        *by = ShellTile<double, s>::BY;         \
        return;
    switch (S) { LBE_BOX(1) LBE_BOX(2) LBE_BOX(3) LBE_BOX(4) LBE_BOX(5) LBE_BOX(6) LBE_BOX(7) default: break; }
#undef LBE_BOX
    *bx = 0;
    *by = 0;
}

}  // namespace lbe
