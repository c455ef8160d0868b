// K3 in FP64 for fields of high contrast: the sums over the half shell, point by point, as e^ [a(r+e) - a(r-e)].
//
// The fixed-point sums (lbe_shell_fixed.cuh) round relative to a field's largest value, this kernel relative to the
// values summed: density over six decades along one axis, diameter 3, error where it is below 1e-4 of its largest, of the
// root of the sum of squares over the shell: 1.3e-14 in fixed point, 1.7e-17 here.  It runs, in place of the
// fixed-point kernel, where some value of a field is 16 times smaller than the field's largest (k_to_fixed sets the
// flag; a value 8 times smaller still has all its 53 bits in fixed point, and up to 16 the two err alike), and only for
// pairs that the FFTs are not the general form of (those err by 6e-13 in the example).
//
// Bound by the FP64 pipe (two lanes per SM): one output per thread, a march through z with the 2S + 1 planes in use in
// shared memory.  256x64x64 of diameters 4 and 6: 11.06 ms, against 0.86 in fixed point (the same sums in one launch per
// pair: 10.70); of diameter 3 0.87 ms, against 0.12.  All pairs in one launch; a launch that finds the flag unset returns
// at once (a step of a 24^3 lattice of diameter 3: 36.4 -> 39.3 us).
#include <algorithm>
#include <utility>

#include "lbe_device.cuh"
#include "lbe_launch.h"
#include "lbe_march.cuh"
#include "lbe_shell.cuh"
#include "lbe_shell_fixed.cuh"

namespace lbe {

// Rows of a tile: the ring of 2S + 2 planes of two fields has to fit shared memory.
__host__ __device__ constexpr int wide_rows(int smax) { return smax >= 5 ? 4 : 8; }

template <int S, int TY>
struct WideTile {
    static constexpr int BX = (32 + 2 * S + 2) / 2 * 2;  // one column of slack for the 16-byte boundary
    static constexpr int BY = TY + 2 * S;
    static constexpr int R = 2 * S + 2;  // ring slots: the planes in use and one in flight
    static constexpr int PLANE = BX * BY;
    static constexpr int PLANE_BYTES = (PLANE * 8 + 127) / 128 * 128;
    static constexpr int SLOT_BYTES = 2 * PLANE_BYTES;
    static constexpr int BYTES = 128 + R * SLOT_BYTES + 128;  // barriers, ring, alignment
};

// Whether e is the listed one of the two points e, -e.
__host__ __device__ constexpr bool positive_half(int x, int y, int z) {
    return z > 0 || (z == 0 && (y > 0 || (y == 0 && x > 0)));
}
template <int S, int BX, int GN, int K>
__device__ __forceinline__ void wide_term(const double *const *sb, double (&an)[3], double (&ag)[3]) {
    constexpr int W = 2 * S + 1, ex = K % W - S, ey = K / W % W - S, ez = K / (W * W);
    if constexpr (in_shell(S, ex, ey, ez) && positive_half(ex, ey, ez)) {
        constexpr double len = ct_sqrt((double)(ex * ex + ey * ey + ez * ez));
        constexpr int off = ey * BX + ex;
        const double *pp = sb[S + ez] + off, *pm = sb[S - ez] - off;
        const double dn = pp[0] - pm[0], dg = pp[GN] - pm[GN];
        constexpr double u[3] = {ex / len, ey / len, ez / len};
        if constexpr (ex != 0) {
            an[0] += u[0] * dn;
            ag[0] += u[0] * dg;
        }
        if constexpr (ey != 0) {
            an[1] += u[1] * dn;
            ag[1] += u[1] * dg;
        }
        if constexpr (ez != 0) {
            an[2] += u[2] * dn;
            ag[2] += u[2] * dg;
        }
    }
}
template <int S, int BX, int GN, int... K>
__device__ __forceinline__ void wide_sum(const double *const *sb, double (&an)[3], double (&ag)[3],
                                         std::integer_sequence<int, K...>) {
    (wide_term<S, BX, GN, K>(sb, an, ag), ...);
}

// Pair (a, b) of the block's tile and planes; the barriers are fresh and every thread takes part.
template <int SMAX, int S>
__device__ __forceinline__ bool wide_march(const ShellMarchMaps &maps, const FixedArgs &A, unsigned char *ring,
                                           uint64_t *bars, int a, int b, int z0, int nout, bool accumulate) {
    constexpr int TY = wide_rows(SMAX);
    using Tl = WideTile<S, TY>;
    const Grid &g = A.g;
    const int tid = threadIdx.x, tx = tid & 31, ty = tid >> 5;
    const int nbx = (g.nx + 31) / 32;
    const int x0 = blockIdx.x % nbx * 32, y0 = blockIdx.x / nbx * TY;
    const int pair = a * A.M + b, nplanes = nout + 2 * S, ox = (g.H - S) & 1;
    const bool leader = tid == 0;
    auto issue = [&](int j) {  // plane j holds interior z = z0 - S + j
        const int slot = j % Tl::R;
        unsigned char *dst = ring + slot * Tl::SLOT_BYTES;
        const int bx = x0 + g.H - S - ox, by = y0 + g.H - S, zp = z0 - S + j + g.H;
        mbar_arrive_expect_tx(&bars[slot], 2u * Tl::PLANE * 8u);
        tma_load_3d(dst, &maps.n[pair], bx, by, zp, &bars[slot]);
        tma_load_3d(dst + Tl::PLANE_BYTES, &maps.gn[pair], bx, by, zp, &bars[slot]);
    };
    if (leader) {
        fence_proxy_async_smem();  // the ring may have been read for the pair before
        for (int j = 0; j < 2 * S + 1 && j < nplanes; ++j) issue(j);
    }
    for (int j = 0; j < 2 * S; ++j)
        if (!mbar_wait_bounded(&bars[j % Tl::R], (uint32_t)(j / Tl::R) & 1u, A.err)) {
            mbar_drain(bars, Tl::R, j, min(2 * S + 1, nplanes));
            return false;
        }
    const int x = x0 + tx, y = y0 + ty;
    const bool active = x < g.nx && y < g.ny;
    const int toff = (ty + S) * Tl::BX + tx + S + ox;
    for (int iz = 0; iz < nout; ++iz) {
        const int jn = iz + 2 * S;
        if (leader && jn + 1 < nplanes) {
            fence_proxy_async_smem();
            issue(jn + 1);
        }
        if (!mbar_wait_bounded(&bars[jn % Tl::R], (uint32_t)(jn / Tl::R) & 1u, A.err)) {
            mbar_drain(bars, Tl::R, jn, min(jn + 2, nplanes));
            return false;
        }
        if (active) {
            const double *sb[2 * S + 1];
#pragma unroll
            for (int k = 0; k <= 2 * S; ++k)
                sb[k] = reinterpret_cast<const double *>(ring + (iz + k) % Tl::R * Tl::SLOT_BYTES) + toff;
            double an[3] = {0, 0, 0}, ag[3] = {0, 0, 0};
            wide_sum<S, Tl::BX, Tl::PLANE_BYTES / 8>(
                sb, an, ag, std::make_integer_sequence<int, (2 * S + 1) * (2 * S + 1) * (S + 1)>{});
            const int z = z0 + iz;
            const long long i = (long long)x + (long long)g.nx * ((long long)y + (long long)g.ny * z);
            const double pre = A.coef[pair] * A.npad[(long long)a * g.P + pidx(g, x, y, z)];
            const double gr = A.gab[(long long)pair * g.N + i];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const double v = pre * (0.5 * gr * an[c] + 0.5 * ag[c]);
                double *o = A.C + (3 * (long long)a + c) * g.N + i;
                *o = accumulate ? *o + v : v;
                if (A.Pout) A.Pout[(3 * (long long)A.q[pair] + c) * g.N + i] = an[c];
            }
        }
        __syncthreads();
    }
    return true;
}

template <int SMAX>
__global__ void __launch_bounds__(32 * wide_rows(SMAX))
    k_shell_wide(const __grid_constant__ ShellMarchMaps maps, const __grid_constant__ FixedArgs A) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char *base = smem_align128(smem_raw);
    uint64_t *bars = reinterpret_cast<uint64_t *>(base);
    pdl_wait();
    if (*A.wide == 0u) return;
    const int a = blockIdx.z / A.nzb, z0 = (blockIdx.z - a * A.nzb) * A.lz;
    const int nout = min(A.lz, A.g.nz - z0);
    bool accumulate = false;
    for (int b = 0; b < A.M; ++b) {
        const int S = A.S[a * A.M + b];
        if (S == 0) continue;
        // the pairs' rings differ: fresh barriers for each (every copy of the pair before was waited for)
        if (threadIdx.x == 0) {
            for (int r = 0; r < 2 * SMAX + 2; ++r) {
                if (accumulate) mbar_inval(&bars[r]);
                mbar_init(&bars[r], 1);
            }
            fence_mbar_init();
        }
        __syncthreads();
        bool ok = true;
        [&]<int... I>(std::integer_sequence<int, I...>) {
            (
                [&] {
                    if (S == I + 1)
                        ok = wide_march<SMAX, I + 1>(maps, A, base + 128, bars, a, b, z0, nout, accumulate);
                }(),
                ...);
        }(std::make_integer_sequence<int, SMAX>{});
        if (!ok) return;
        accumulate = true;
    }
}

template <int SMAX>
static cudaError_t launch_wide_t(int Smax, const ShellMarchMaps &maps, FixedArgs &A, cudaStream_t st) {
    constexpr int TY = wide_rows(SMAX);
    static PerDevice once;
    const cudaError_t e = allow_smem(once, k_shell_wide<SMAX>, WideTile<SMAX, TY>::BYTES);
    if (e != cudaSuccess) return e;
    int smem = 0;  // of the launch's widest shell
    [&]<int... I>(std::integer_sequence<int, I...>) {
        ((smem = Smax == I + 1 ? WideTile<I + 1, TY>::BYTES : smem), ...);
    }(std::make_integer_sequence<int, SMAX>{});
    const Grid &g = A.g;
    const int most = 65535 / A.M;
    A.lz = std::max(16, (g.nz + most - 1) / most);
    A.nzb = (g.nz + A.lz - 1) / A.lz;
    const int tiles = (g.nx + 31) / 32 * ((g.ny + TY - 1) / TY);
    return launch_pdl(k_shell_wide<SMAX>, dim3(tiles, 1, A.M * A.nzb), 32 * TY, smem, st, maps, A);
}
cudaError_t launch_shell_wide(int Smax, const ShellMarchMaps &maps, FixedArgs &A, cudaStream_t st) {
    if (Smax < 1 || Smax > 7) return cudaErrorInvalidValue;
    return Smax <= 4 ? launch_wide_t<4>(Smax, maps, A, st) : launch_wide_t<7>(Smax, maps, A, st);
}

void shell_wide_box(int Smax, int S, int *bx, int *by) {
    *bx = (32 + 2 * S + 2) / 2 * 2;
    *by = wide_rows(Smax) + 2 * S;
}

}  // namespace lbe
