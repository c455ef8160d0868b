// Dispatch of the shell-force kernels by precision and pair diameter, and the host-side shell helpers.
// FP32: every pair in one launch of the marching kernel (lbe_shell_march.cuh), instantiated for the largest
// pair diameter 4, 6 or 8 (the registers of a thread grow with it: 128, 162, 206, so four, three and two
// blocks of 128 threads per SM).  FP64: the same march in fixed point (lbe_shell_fixed.cuh) on the integer images
// of the padded fields that k_to_fixed writes.
#include "lbe_device.cuh"
#include "lbe_launch.h"
#include "lbe_shell.cuh"
#include "lbe_shell_fixed.cuh"
#include "lbe_shell_march.cuh"

namespace lbe {

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

cudaError_t launch_shell_fixed_4(const ShellMarchMaps &maps, FixedArgs &A, cudaStream_t st);
cudaError_t launch_shell_fixed_6(const ShellMarchMaps &maps, FixedArgs &A, cudaStream_t st);
cudaError_t launch_shell_fixed_7(const ShellMarchMaps &maps, FixedArgs &A, cudaStream_t st);

cudaError_t launch_shell_fixed(int Smax, const ShellMarchMaps &maps, FixedArgs &A, cudaStream_t st) {
    if (Smax < 1 || Smax > 7) return cudaErrorInvalidValue;
    return Smax <= 4 ? launch_shell_fixed_4(maps, A, st)
                     : (Smax <= 6 ? launch_shell_fixed_6(maps, A, st) : launch_shell_fixed_7(maps, A, st));
}

// Fixed-point image of a field: v 2^(bits - 1 - e), e the exponent of the field's largest value, rounded to
// nearest, by shifts of the mantissa (no FP64 operation).  Zero, subnormal and non-finite values become 0 (a
// non-finite density is an error of its own).
__device__ __forceinline__ long long to_fixed(double v, int top, int bits) {
    const long long b = __double_as_longlong(v);
    const int e = (int)((b >> 52) & 0x7ff);
    if (e == 0 || e == 0x7ff || top == 0 || top == 0x7ff || e > top) return 0;
    const long long m = (b & 0xfffffffffffffll) | 0x10000000000000ll;
    const int d = top - e - (bits - 53);  // right shift
    const long long r = d <= 0 ? m << -d : (d > 54 ? 0 : (m + (1ll << (d - 1))) >> d);
    return b < 0 ? -r : r;
}
// Whether a value lies so far below the field's largest (a factor of 8 to 16) that the image may drop some of its bits.
__device__ __forceinline__ bool far_below(double v, int top) {
    const long long b = __double_as_longlong(v);
    const int e = (int)((b >> 52) & 0x7ff);
    return (b << 1) != 0 && (e + 3 < top || e == 0);
}
__global__ void __launch_bounds__(256) k_to_fixed(const double *__restrict__ npad, const double *__restrict__ gnpad,
                                                 long long P, int M, int bits, const unsigned *__restrict__ top,
                                                 unsigned *__restrict__ wide, long long *__restrict__ out) {
    pdl_wait();
    bool low = false;
    const int f = blockIdx.y;  // n_b, then g_ab n_b
    const double *src = f < M ? npad + f * P : gnpad + (long long)(f - M) * P;
    const int e = fx_exponent(top[f]);
    longlong2 *dst = reinterpret_cast<longlong2 *>(out + f * P);
    const double2 *s2 = reinterpret_cast<const double2 *>(src);
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < P / 2;
         i += (long long)gridDim.x * blockDim.x) {
        const double2 v = s2[i];
        dst[i] = make_longlong2(to_fixed(v.x, e, bits), to_fixed(v.y, e, bits));
        low = low || far_below(v.x, e) || far_below(v.y, e);
    }
    // (wide: NULL where nothing asks; most warps find the word set already)
    if (wide && __any_sync(0xffffffffu, low) && (threadIdx.x & 31) == 0 && *(volatile unsigned *)wide == 0u) *wide = 1u;
}
cudaError_t launch_to_fixed(int Smax, const double *npad, const double *gnpad, long long P, int M,
                            const unsigned *top, unsigned *wide, long long *out, cudaStream_t st) {
    const long long nb = (P / 2 + 255) / 256;
    return launch_pdl(k_to_fixed, dim3((unsigned)(nb < 2048 ? nb : 2048), M + M * M), 256, 0, st, npad, gnpad, P, M,
                      fx_bits(Smax), top, wide, out);
}

bool shell_supported(bool fp64, int S) { return S >= 1 && S <= (fp64 ? 7 : 8); }

// Box of the shell-transpose tiles (lbe_adj_shell.cuh, dispatched in lbe_adjoint.cu).  FP32: the
// interleaved 8-byte (Lambda, g Lambda) elements of a 32 x 16 tile (32 x 8 at S = 8), the tile the
// transpose itself runs; FP64: two separate planes of a 32 x 8 tile (32 x 4 from S = 5).
void adj_shell_box(bool fp64, int S, int *bx, int *by) {
    if (!fp64) {
        *bx = ((32 + 2 * S + 1) + 1) / 2 * 2;
        *by = (S <= 7 ? 16 : 8) + 2 * S;
        return;
    }
    *bx = ((32 + 2 * S + 1) + 1) / 2 * 2;  // ShellTileZ<double, S, 1, .>
    *by = (S >= 5 ? 4 : 8) + 2 * S;
}

double shell_march_cost(bool fp64, const Grid &g, int M, int Smax, bool swap) {
    const MarchAxes dir = march_axes(g, swap);
    const int ty = fp64 ? FX_TY : SM_TY;
    const int smax = Smax <= 4 ? 4 : (Smax <= 6 ? 6 : (fp64 ? 7 : 8));
    const int per_sm = fp64 ? fixed_per_sm(smax) : shell_march_per_sm(smax);
    const long long tiles = (long long)((g.nx + 31) / 32) * ((dir.rows + ty - 1) / ty);
    double cost = 0.0;
    march_planes(tiles * M, dir.planes, smax, per_sm, 1.0, 0.9, M > 1, 65535 / M, &cost);
    return cost;
}

void shell_box(bool fp64, int S, int *bx, int *by) {
    if (!fp64) {  // ShellMarchTile
        *bx = 32 + 2 * ((S + 3) / 4 * 4);
        *by = SM_TY + 2 * S;
        return;
    }
    *bx = 32 + 2 * ((S + 1) / 2 * 2);  // FixedTile
    *by = FX_TY + 2 * S;
}

}  // namespace lbe
