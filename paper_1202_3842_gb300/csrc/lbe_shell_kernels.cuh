// Kernel template of the FP64 mean-field shell force (K3) and its launcher.
// Included by the translation units that instantiate them (one group of pair
// diameters each, so the builds run in parallel).
//
// K3 in FP64: mean-field Enskog force of one ordered species pair (a, b) (Appendix,
// hard-sphere C^{alpha,mf}):
//   C^a(r) (+)= -kT sigma_ab^2 w_ab n_a(r) sum_{e in K_ab} e^ (g_ab(r) + g_ab(r+e))/2 n_b(r+e)
//            =  coef * n_a(r) * [ g_ab(r)/2 * sum e^ n_b(r+e) + 1/2 * sum e^ (g_ab n_b)(r+e) ]
// with coef = -kT sigma_ab^2 w_ab.  Both sums run over the half shell as
// e^ [a(r+e) - a(r-e)].
//
// Data path: the padded fields are streamed plane by plane (z-marching) into a
// shared-memory ring by TMA (cp.async.bulk.tensor, 2-D boxes of
// (32 + 2S) x (TY + 2S) per plane, completion on an mbarrier per ring slot).
// The kernel (FP64; FP32 runs lbe_shell_march.cuh) reads the padded density n_b and the padded product
// g_ab*n_b as two planes and gives each thread one output per plane.  The shell offsets and unit vectors are
// compile-time immediates.  When Pout is given, the kernel also stores
// P = sum_e e^ n_b(r+e) of the pair ([3][N]), which the discrete adjoint needs.
#pragma once
#include <utility>

#include "lbe_device.cuh"
#include "lbe_launch.h"
#include "lbe_march.cuh"
#include "lbe_shell.cuh"

namespace lbe {

template <int S>
struct ShellTable {
    static constexpr auto hs = make_half_shell<S>();
    static constexpr int count = half_shell_count(S);
};

template <typename T, int S, int I>
__device__ __forceinline__ void shell_term(const T *const *sb, T *an, T *ag) {
    using Tl = ShellTile<T, S>;
    constexpr int ex = ShellTable<S>::hs.e[I][0];
    constexpr int ey = ShellTable<S>::hs.e[I][1];
    constexpr int ez = ShellTable<S>::hs.e[I][2];
    constexpr double len = ct_sqrt((double)(ex * ex + ey * ey + ez * ez));
    constexpr int off = ey * Tl::BX + ex;
    constexpr int GN = Tl::PLANE_BYTES / (int)sizeof(T);
    const T *pp = sb[S + ez] + off;
    const T *pm = sb[S - ez] - off;
    const T dn = pp[0] - pm[0];
    const T dg = pp[GN] - pm[GN];
    if constexpr (ex != 0) {
        constexpr T u = (T)(ex / len);
        an[0] += u * dn;
        ag[0] += u * dg;
    }
    if constexpr (ey != 0) {
        constexpr T u = (T)(ey / len);
        an[1] += u * dn;
        ag[1] += u * dg;
    }
    if constexpr (ez != 0) {
        constexpr T u = (T)(ez / len);
        an[2] += u * dn;
        ag[2] += u * dg;
    }
}

template <typename T, int S, int... I>
__device__ __forceinline__ void shell_sum(const T *const *sb, T *an, T *ag, std::integer_sequence<int, I...>) {
    (shell_term<T, S, I>(sb, an, ag), ...);
}

template <typename T, int S>
__global__ void __launch_bounds__(32 * ShellTile<T, S>::TY)
    k_shell_force(const __grid_constant__ CUtensorMap map_n, const __grid_constant__ CUtensorMap map_gn,
                  Grid g, int ox, const T *__restrict__ npad_a, const T *__restrict__ g_ab,
                  T *__restrict__ Cout, T *__restrict__ Pout, T coef, int accumulate, int *err) {
    using Tl = ShellTile<T, S>;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *base = smem_align128(smem_raw);
    T *ring = reinterpret_cast<T *>(base);
    uint64_t *bars = reinterpret_cast<uint64_t *>(base + Tl::R * Tl::SLOT_BYTES);
    constexpr int SLOT = Tl::SLOT_BYTES / (int)sizeof(T);

    const int tx = threadIdx.x, ty = threadIdx.y;
    const int x0 = blockIdx.x * Tl::TX, y0 = blockIdx.y * Tl::TY, z0 = blockIdx.z * Tl::LZ;
    const int zend = min(z0 + Tl::LZ, g.nz);
    const int nout = zend - z0;
    const int nplanes = nout + 2 * S;
    const bool leader = (tx == 0 && ty == 0);
    const int bx = x0 + g.H - S - ox;  // multiple of 16 bytes / sizeof(T)
    const int by = y0 + g.H - S;
    constexpr uint32_t tx_bytes = 2u * Tl::PLANE * (uint32_t)sizeof(T);

    if (leader) {
        prefetch_tensormap(&map_n);
        prefetch_tensormap(&map_gn);
        for (int r = 0; r < Tl::R; ++r) mbar_init(&bars[r], 1);
        fence_mbar_init();
    }
    __syncthreads();

    auto issue = [&](int j) {  // plane j holds interior z = z0 - S + j
        const int slot = j % Tl::R;
        unsigned char *dst = base + slot * Tl::SLOT_BYTES;
        const int zp = z0 - S + j + g.H;
        mbar_arrive_expect_tx(&bars[slot], tx_bytes);
        tma_load_3d(dst, &map_n, bx, by, zp, &bars[slot]);
        tma_load_3d(dst + Tl::PLANE_BYTES, &map_gn, bx, by, zp, &bars[slot]);
    };
    if (leader) {
        for (int j = 0; j < 2 * S + 1 && j < nplanes; ++j) issue(j);
    }
    for (int j = 0; j < 2 * S; ++j)
        if (!mbar_wait_bounded(&bars[j % Tl::R], (j / Tl::R) & 1, err)) {
            mbar_drain(bars, Tl::R, j, min(2 * S + 1, nplanes));
            return;
        }

    const int x = x0 + tx, y = y0 + ty;
    const bool active = (x < g.nx) && (y < g.ny);
    const int toff = (ty + S) * Tl::BX + (tx + S + ox);
    const T half = (T)0.5;

    for (int iz = 0; iz < nout; ++iz) {
        if (leader && iz + 2 * S + 1 < nplanes) {
            fence_proxy_async_smem();
            issue(iz + 2 * S + 1);
        }
        const int jn = iz + 2 * S;
        if (!mbar_wait_bounded(&bars[jn % Tl::R], (jn / Tl::R) & 1, err)) {
            mbar_drain(bars, Tl::R, jn, min(iz + 2 * S + 2, nplanes));
            return;
        }
        if (active) {
            const T *sb[2 * S + 1];
#pragma unroll
            for (int k = 0; k <= 2 * S; ++k) sb[k] = ring + ((iz + k) % Tl::R) * SLOT + toff;
            T an[3] = {0, 0, 0}, ag[3] = {0, 0, 0};
            shell_sum<T, S>(sb, an, ag, std::make_integer_sequence<int, ShellTable<S>::count>{});
            const int z = z0 + iz;
            const long long i = (long long)x + (long long)g.nx * ((long long)y + (long long)g.ny * z);
            const T na = npad_a[pidx(g, x, y, z)];
            const T gr = g_ab[i];
            const T pre = coef * na;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const T v = pre * (half * gr * an[c] + half * ag[c]);
                T *o = Cout + (long long)c * g.N + i;
                if (accumulate)
                    *o += v;
                else
                    *o = v;
                if (Pout) Pout[(long long)c * g.N + i] = an[c];
            }
        }
        __syncthreads();
    }
}

template <typename T, int S>
cudaError_t launch_one(const ShellLaunch &L, cudaStream_t st) {
    using Tl = ShellTile<T, S>;
    static bool attr_set = false;
    if (!attr_set) {
        cudaError_t e = cudaFuncSetAttribute(k_shell_force<T, S>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             Tl::SMEM);
        if (e != cudaSuccess) return e;
        attr_set = true;
    }
    const Grid &g = *L.grid;
    dim3 block(Tl::TX, Tl::TY, 1);
    dim3 grid((g.nx + Tl::TX - 1) / Tl::TX, (g.ny + Tl::TY - 1) / Tl::TY, (g.nz + Tl::LZ - 1) / Tl::LZ);
    const int A = Tl::A;
    const int ox = ((g.H - S) % A + A) % A;
    k_shell_force<T, S><<<grid, block, Tl::SMEM, st>>>(*L.map_n, *L.map_gn, g, ox, (const T *)L.npad_a,
                                                       (const T *)L.g_ab, (T *)L.Cout, (T *)L.Pout, (T)L.coef,
                                                       L.accumulate, L.err);
    return cudaGetLastError();
}

}  // namespace lbe
