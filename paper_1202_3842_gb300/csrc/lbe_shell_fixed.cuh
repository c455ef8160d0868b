// K3 in FP64: the marching shell force (lbe_shell_march.cuh: formulas, march, exchange of P) with the shell sums
// in 64-bit fixed point.
//
// GB300 issues two FP64 operations per clock and SM and 64 or more integer ones, so the FP64 sums are bound by
// that pipe (83 ms of the 512x128x128 step point by point; 24 ms as FFTs).  A shell sum is a sum of one field
// with fixed weights, which integers hold exactly:
//   - every field is scaled by a power of two that gives its largest value fx_bits bits, 57 up to diameter 4 and 56
//     beyond (k_to_fixed; the maxima come from K2): values down to an eighth of the largest keep all their 53
//     bits, smaller ones are rounded at 2^-56 of it;
//   - of a plane's points those with X^2 + Y^2 = rho share the weight 1/|e| for a given |Z|: their sums
//     S = sum v, A_x = sum X v, A_y = sum Y v are exact (64-bit adds, small multipliers);
//   - each sum is multiplied once per |Z| by 1/sqrt(rho + Z^2), known to 61 bits, as three 32-bit multiplies
//     that keep the product to about one unit of the fixed point.
// Everything after that is exact again (adds and the factor Z), until the sums of an output become doubles.  The
// result is the sum of the definition to a few 2^-55 of the field's largest value, where FP64 sums (and more so
// the FFTs) round at every addition.  FP64 sums round relative to the values at hand, though: where a field's
// values lie more than a factor of 8 to 16 apart, k_shell_wide takes the launch (lbe_shell_wide.cu), except for
// pairs whose general form are the FFTs, which round relative to the whole field, ten times as much.
// Error of C against sums in extended precision, rms over max |C| (300 nodes; this kernel, the FP64 stencil it
// replaces, the FFTs that were the default from diameter 4 on): 24^3 with 1% noise, diameter 3 9.0e-16, 9.2e-16,
// 8.4e-15; diameter 6 1.15e-15, 1.08e-15, 1.3e-14; diameter 7 1.5e-15, 1.3e-15, 1.2e-14; 48^3 well of diameter 6
// after 50 steps 2.65e-16, 2.61e-16, 3.3e-16; 48x24x24 channel of diameters 4 and 6 6.5e-16, 6.6e-16, 6.8e-16.
//
// Shell stage on GB300: 256x64x64 channel of diameters 4 and 6 12.2 ms (stencil) and 3.12 ms (FFTs) -> 0.86 ms;
// 48^3 well of diameter 4 114 us (FFTs) -> 46; 24^3 well of diameter 3 429 us (stencil, six blocks) -> 16;
// 512x512x1 of diameter 6 265 us (FFTs) -> 190, along y.
// At diameter 6 a warp takes 1400 instructions for 32 outputs of one field and plane; the integer pipe is busy
// half of the cycles at 2.6 warps per scheduler, the rest is latency of the multiply chains.
//
// One output and one field per thread: the running sums take 12 S registers, the plane's B about 60 at S = 6.  Where the
// largest diameter is 5 or 6, the 168 registers of three blocks per SM do not hold them all (288 bytes of spill stores and
// 148 of loads in the code); up to 4 and at 7 nothing spills.
#pragma once
#include "lbe_launch.h"
#include "lbe_march.cuh"

namespace lbe {

// Bits of a field's largest value: as many as the ring sums of the launch's widest shell leave room for.
__host__ __device__ constexpr int fx_bits(int smax) { return smax <= 4 ? 57 : 56; }
constexpr int FX_TY = 2;   // output rows of a tile (32 x FX_TY outputs per plane)
constexpr int FX_R = 4;    // ring slots

using i64 = long long;
using u64 = unsigned long long;

// floor(2^61 / sqrt(d)), or 2^60 / sqrt(d) for the shell of diameter 1 (whose largest weight is 1): the weight's
// bits; a product with it is in units of 2^fx_unit(S) of the fixed point.
__host__ __device__ constexpr int fx_unit(int S) { return S == 1 ? 2 : 1; }
__host__ __device__ constexpr u64 fx_weight(int S, int d) {
    const int bits = 62 - fx_unit(S);
    u64 lo = 0, hi = 1ull << bits;  // largest w with w^2 d <= 2^(2 bits)
    while (lo < hi) {
        const u64 m = lo + (hi - lo + 1) / 2;
        if ((unsigned __int128)m * m <= ((unsigned __int128)1 << (2 * bits)) / (unsigned)d)
            lo = m;
        else
            hi = m - 1;
    }
    return lo;
}
// The weight as wh 2^30 + wl, |wl| <= 2^29.
__host__ __device__ constexpr int fx_wh(int S, int d) { return (int)((fx_weight(S, d) + (1ull << 29)) >> 30); }
__host__ __device__ constexpr int fx_wl(int S, int d) { return (int)((i64)fx_weight(S, d) - ((i64)fx_wh(S, d) << 30)); }

__host__ __device__ constexpr bool ring_has(int S, int rho) {  // some (X, Y) of the shell's projection has X^2 + Y^2 = rho
    for (int x = 0; x <= S; ++x)
        for (int y = 0; y <= S; ++y)
            if (x * x + y * y == rho && ring_mask(S, x, y)) return true;
    return false;
}
// Sum of X over the ring's points with X > 0 (of all points with rho = 0 or for c = 2: their number): the ring
// sum's bound in units of the field's.
__host__ __device__ constexpr int ring_weight(int S, int rho, int c) {
    int n = 0;
    for (int x = -S; x <= S; ++x)
        for (int y = -S; y <= S; ++y)
            if (x * x + y * y == rho) n += c == 2 ? 1 : (x > 0 ? x : 0);
    return n;
}
__host__ __device__ constexpr bool fx_term(int S, int rho, int Z) {
    return rho + Z * Z >= S * S - S + 1 && rho + Z * Z <= S * S + S && ring_has(S, rho);
}
// Bounds that the arithmetic below rests on, checked for every diameter:
// - (ring sum) >> 30 fits 32 bits; the low products of one B fit 32 bits around FX_OFF.
constexpr u64 FX_OFF = 1ull << 30;
__host__ __device__ constexpr bool fx_bounds_hold(int S, int bits) {
    for (int c = 0; c < 3; c += 2)
        for (int Z = 0; Z <= S; ++Z) {
            u64 up = 0, down = 0;  // of the sum of (al wh + a30 wl) >> 32
            for (int rho = 0; rho <= S * S + S; ++rho) {
                if (!fx_term(S, rho, Z)) continue;
                const u64 A = (u64)ring_weight(S, rho, c) << bits;
                if (A >= (1ull << 61)) return false;
                const int wl = fx_wl(S, rho + Z * Z);
                const u64 low = (u64)(((unsigned __int128)(A >> 30) * (u64)(wl < 0 ? -wl : wl)) >> 32) + 1;
                if (fx_wh(S, rho + Z * Z) > (1 << 30) + (1 << 29)) return false;  // al wh + a30 wl fits 63 bits
                up += (u64)fx_wh(S, rho + Z * Z) + low;
                down += low;
            }
            if (down >= FX_OFF || up + FX_OFF >= (1ull << 32)) return false;
        }
    return true;
}

// - an output's whole sum, in units of 2^fx_unit, fits 63 bits.
__host__ __device__ constexpr bool fx_sum_fits(int S, int bits) {
    int x = 0;  // sum of e_x over the shell's points with e_x > 0, above sum e_x / |e| times S
    for (int X = 1; X <= S; ++X)
        for (int Y = -S; Y <= S; ++Y)
            for (int Z = -S; Z <= S; ++Z)
                if (in_shell(S, X, Y, Z)) x += X;
    // |e| >= S - 1/2
    return ((unsigned __int128)(unsigned)x << bits) / (unsigned)(2 * S - 1) * 2 >> fx_unit(S) < ((u64)1 << 63);
}

template <int S>
struct FixedTile {
    static constexpr int S2 = (S + 1) / 2 * 2;  // halo along x: keeps the copies on 16-byte boundaries
    static constexpr int BX = 32 + 2 * S2;
    static constexpr int BY = FX_TY + 2 * S;
    static constexpr int PLANE = BX * BY;
    static constexpr int PLANE_BYTES = (PLANE * 8 + 127) / 128 * 128;
    static constexpr int SLOT_BYTES = 2 * PLANE_BYTES;
};
__host__ __device__ constexpr int fixed_per_sm(int smax) { return smax <= 6 ? 3 : 2; }
template <int SMAX>
struct FixedSmem {
    static constexpr int SLOT = FixedTile<SMAX>::SLOT_BYTES;
    static constexpr int XCH = FX_R * SLOT;  // P exchange: [2][3][32 FX_TY] doubles
    static constexpr int BARS = XCH + 2 * 3 * 32 * FX_TY * 8;
    static constexpr int BYTES = BARS + FX_R * 8 + 128;
};

__device__ __forceinline__ i64 mad_wide(int a, int b, i64 c) {
    i64 d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}
__device__ __forceinline__ i64 mad_wide_u(unsigned a, unsigned b, i64 c) {
    i64 d;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}

// B of one component and height: the sum over rings of A W 2^-62, W = WH 2^30 + WL.  Of the product's parts, A_hi WH
// is whole; the other two are summed with half a unit before their 32 low bits are dropped, so the rounding has no
// bias and a ring sum of 0 adds exactly 0.
struct FixedSum {
    i64 hi = 0;
    unsigned lo = (unsigned)FX_OFF;
    template <int WH, int WL>
    __device__ __forceinline__ void add(i64 A) {
        hi = mad_wide((int)(A >> 32), WH, hi);
        const i64 t = mad_wide((int)(A >> 30), WL, mad_wide_u((unsigned)A, (unsigned)WH, 1ll << 31));
        lo += (unsigned)(t >> 32);
    }
    __device__ __forceinline__ i64 value() const { return hi + ((i64)(u64)lo - (i64)FX_OFF); }
};

template <int S, int BX, int RHO>
__device__ __forceinline__ void fixed_ring(const i64 *c, FixedSum *Bx, FixedSum *By, FixedSum *Bz) {
    if constexpr (ring_has(S, RHO)) {
        i64 s = 0, ax = 0, ay = 0;
        [&]<int... K>(std::integer_sequence<int, K...>) {
            (
                [&] {
                    constexpr int X = K / (S + 1), Y = K % (S + 1);
                    if constexpr (X * X + Y * Y == RHO) {
                        if constexpr (X == 0 && Y == 0) {
                            s += c[0];
                        } else if constexpr (X == 0) {
                            const i64 a = c[Y * BX], d = c[-Y * BX];
                            s += a + d;
                            ay += (i64)Y * (a - d);
                        } else if constexpr (Y == 0) {
                            const i64 a = c[X], b = c[-X];
                            s += a + b;
                            ax += (i64)X * (a - b);
                        } else {
                            const i64 a = c[Y * BX + X], b = c[Y * BX - X];
                            const i64 cc = c[-Y * BX + X], d = c[-Y * BX - X];
                            const i64 u = a - d, v = cc - b;
                            s += a + d + b + cc;
                            ax += (i64)X * (u + v);
                            ay += (i64)Y * (u - v);
                        }
                    }
                }(),
                ...);
        }(std::make_integer_sequence<int, (S + 1) * (S + 1)>{});
        [&]<int... ZI>(std::integer_sequence<int, ZI...>) {
            (
                [&] {
                    constexpr int Z = ZI;
                    if constexpr (fx_term(S, RHO, Z)) {
                        constexpr int WH = fx_wh(S, RHO + Z * Z), WL = fx_wl(S, RHO + Z * Z);
                        if constexpr (RHO > 0) {
                            Bx[Z].template add<WH, WL>(ax);
                            By[Z].template add<WH, WL>(ay);
                        }
                        if constexpr (Z > 0) Bz[Z].template add<WH, WL>(s);
                    }
                }(),
                ...);
        }(std::make_integer_sequence<int, S + 1>{});
    }
}
template <int S, int BX, int... RHO>
__device__ __forceinline__ void fixed_plane(const i64 *c, FixedSum *Bx, FixedSum *By, FixedSum *Bz,
                                            std::integer_sequence<int, RHO...>) {
    (fixed_ring<S, BX, RHO>(c, Bx, By, Bz), ...);
}

struct FixedArgs {
    Grid g;
    MarchAxes dir;
    int M, lz, nzb;
    int order[MAXS];
    int S[MAXS * MAXS], q[MAXS * MAXS];
    double coef[MAXS * MAXS];
    const unsigned *top;  // high words of the fields' largest values: n_b [M], g_ab n_b [M][M]
    const unsigned *wide; // NULL, or not 0 where a field's values lie too far apart: k_shell_wide takes the pairs
    const double *npad, *gab;
    double *C, *Pout;
    int *err;
};

// Exponent of a field's largest value from its high word (0 if it is not a normal number: the field is 0 then).
__device__ __forceinline__ int fx_exponent(unsigned top) { return (int)((top >> 20) & 0x7ffu); }
// 2^(k) as a double, k clamped to the normal range.
__device__ __forceinline__ double fx_pow2(int k) {
    k = max(-1022, min(1023, k));
    return __hiloint2double((1023 + k) << 20, 0);
}

template <int SMAX, int S>
__device__ __forceinline__ bool fixed_march(const ShellMarchMaps &maps, const FixedArgs &A, unsigned char *base,
                                            uint64_t *bars, int a, int b, int z0, int nout, bool accumulate, int &it) {
    static_assert(fx_bounds_hold(S, fx_bits(SMAX)) && fx_sum_fits(S, fx_bits(SMAX)), "fixed-point ranges");
    using Tl = FixedTile<S>;
    using Sm = FixedSmem<SMAX>;
    const Grid &g = A.g;
    const MarchAxes &dir = A.dir;
    const int tid = threadIdx.x;
    const int fld = tid / (32 * FX_TY);  // 0: P (n_b), 1: Q (g_ab n_b)
    const int ot = tid - fld * (32 * FX_TY);
    const int row = ot >> 5, tx = ot & 31;
    const int nbx = (g.nx + 31) / 32;  // tiles of a plane lie along the grid's x, which has room for all
    const int x0 = blockIdx.x % nbx * 32, y0 = blockIdx.x / nbx * FX_TY;
    const int x = x0 + tx, y = y0 + row;
    const int pair = a * A.M + b;
    const int nplanes = nout + 2 * S;
    const bool leader = tid == 0;
    const int first_it = it;
    double *xch = reinterpret_cast<double *>(base + Sm::XCH);

    auto issue = [&](int j) {  // plane j holds interior z = z0 - S + j (z: along the march, y: along the rows)
        const int k = first_it + j, slot = k % FX_R;
        unsigned char *dst = base + slot * Sm::SLOT;
        const int bx = x0 + g.H - Tl::S2, by = y0 + g.H - S, zp = z0 - S + j + g.H;
        mbar_arrive_expect_tx(&bars[slot], 2u * Tl::PLANE * 8u);
        tma_load_3d(dst, &maps.n[pair], bx, dir.swap ? zp : by, dir.swap ? by : zp, &bars[slot]);
        tma_load_3d(dst + Tl::PLANE_BYTES, &maps.gn[pair], bx, dir.swap ? zp : by, dir.swap ? by : zp, &bars[slot]);
    };
    if (leader) {
        if (first_it > 0) fence_proxy_async_smem();  // the ring was read for the pair before
        for (int j = 0; j < FX_R && j < nplanes; ++j) issue(j);
    }

    i64 ax[2 * S], ay[2 * S], az[2 * S];
#pragma unroll
    for (int k = 0; k < 2 * S; ++k) ax[k] = ay[k] = az[k] = 0;
    const bool act = x < g.nx && y < dir.rows;
    unsigned i = (unsigned)x + dir.srow * (unsigned)y + dir.splane * (unsigned)z0;
    // fixed point to double: the field's scale, and the unit of the products
    const int top = fx_exponent(A.top[fld == 0 ? b : A.M + pair]);
    const double unit = fx_pow2(top - 1023 - (fx_bits(SMAX) - 1) + fx_unit(S));
    const double half_coef = 0.5 * A.coef[pair];
    double *const Ca = A.C + 3 * (long long)a * g.N, *const Pa = A.Pout ? A.Pout + 3 * (long long)A.q[pair] * g.N : nullptr;
    const long long comp[3] = {0, march_component(g, dir, 1), march_component(g, dir, 2)};
    const double *gb = A.gab + (long long)pair * g.N;
    const double *np = A.npad + (long long)a * g.P + march_pidx(g, dir, x, y, z0);
    const int coff = (row + S) * Tl::BX + tx + Tl::S2;

    double na = 0.0, gr = 0.0, old[3] = {0.0, 0.0, 0.0};  // the epilogue's reads, one plane ahead
    auto load_epilogue = [&] {
        na = *np;
        if (fld == 0) {
            gr = gb[i];
        } else if (accumulate) {
#pragma unroll
            for (int c = 0; c < 3; ++c) old[c] = Ca[comp[c] + i];
        }
    };
    if (act) load_epilogue();

    for (int j = 0; j < nplanes; ++j) {
        const int k = first_it + j, slot = k % FX_R;
        if (!mbar_wait_bounded(&bars[slot], (uint32_t)(k / FX_R) & 1u, A.err)) {
            mbar_drain(bars, FX_R, k, first_it + min(j + FX_R, nplanes));
            return false;
        }
        const bool out = j >= 2 * S && act;
        FixedSum Bx[S + 1], By[S + 1], Bz[S + 1];
        const i64 *c = reinterpret_cast<const i64 *>(base + slot * Sm::SLOT + fld * Tl::PLANE_BYTES) + coff;
        fixed_plane<S, Tl::BX>(c, Bx, By, Bz, std::make_integer_sequence<int, S * S + S + 1>{});
        i64 bx[S + 1], by[S + 1], bz[S + 1];
#pragma unroll
        for (int Z = 0; Z <= S; ++Z) {
            bx[Z] = Bx[Z].value();
            by[Z] = By[Z].value();
            bz[Z] = Z > 0 ? Z * Bz[Z].value() : 0;
        }
        const i64 v[3] = {ax[0] + bx[S], ay[0] + by[S], az[0] + bz[S]};
#pragma unroll
        for (int o = 1; o < 2 * S; ++o) {
            const int Z = o < S ? S - o : o - S;
            ax[o - 1] = ax[o] + bx[Z];
            ay[o - 1] = ay[o] + by[Z];
            az[o - 1] = o < S ? az[o] + bz[Z] : az[o] - bz[Z];
        }
        ax[2 * S - 1] = bx[S];
        ay[2 * S - 1] = by[S];
        az[2 * S - 1] = -bz[S];
        double *xo = xch + (j & 1) * (3 * 32 * FX_TY) + ot;
        const double pre = na * half_coef;
        if (fld == 0 && out) {
            const double gp = pre * gr;
#pragma unroll
            for (int cc = 0; cc < 3; ++cc) {
                const double p = unit * (double)v[cc];
                xo[cc * (32 * FX_TY)] = gp * p;
                if (Pa) Pa[comp[cc] + i] = p;
            }
        }
        __syncthreads();
        if (leader && j + FX_R < nplanes) {
            fence_proxy_async_smem();
            issue(j + FX_R);
        }
        if (fld == 1 && out) {
#pragma unroll
            for (int cc = 0; cc < 3; ++cc)
                Ca[comp[cc] + i] = old[cc] + fma(pre, unit * (double)v[cc], xo[cc * (32 * FX_TY)]);
        }
        if (j >= 2 * S) {
            i += dir.splane;
            np += dir.pplane;
            if (act && j + 1 < nplanes) load_epilogue();
        }
    }
    it = first_it + nplanes;
    return true;
}

template <int SMAX>
__global__ void __launch_bounds__(64 * FX_TY, fixed_per_sm(SMAX))
    k_shell_fixed(const __grid_constant__ ShellMarchMaps maps, const __grid_constant__ FixedArgs A) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char *base = smem_align128(smem_raw);
    uint64_t *bars = reinterpret_cast<uint64_t *>(base + FixedSmem<SMAX>::BARS);
    const int k = blockIdx.z / A.nzb, a = A.order[k];
    const int z0 = (blockIdx.z - k * A.nzb) * A.lz;
    const int nout = min(A.lz, A.dir.planes - z0);
    if (threadIdx.x == 0) {
        for (int r = 0; r < FX_R; ++r) mbar_init(&bars[r], 1);
        fence_mbar_init();
    }
    __syncthreads();
    pdl_wait();
    if (nout <= 0 || (A.wide && *A.wide)) return;
    int it = 0;
    bool accumulate = false;
    for (int b = 0; b < A.M; ++b) {
        const int S = A.S[a * A.M + b];
        if (S == 0) continue;
        bool ok = true;
        [&]<int... I>(std::integer_sequence<int, I...>) {
            (
                [&] {
                    if (S == I + 1)
                        ok = fixed_march<SMAX, I + 1>(maps, A, base, bars, a, b, z0, nout, accumulate, it);
                }(),
                ...);
        }(std::make_integer_sequence<int, SMAX>{});
        if (!ok) return;
        accumulate = true;
    }
}

template <int SMAX>
cudaError_t launch_shell_fixed_t(const ShellMarchMaps &maps, FixedArgs &A, cudaStream_t st) {
    constexpr int smem = FixedSmem<SMAX>::BYTES;
    static PerDevice once;
    const cudaError_t e = allow_smem(once, k_shell_fixed<SMAX>, smem);
    if (e != cudaSuccess) return e;
    const Grid &g = A.g;
    const int tiles = (g.nx + 31) / 32 * ((A.dir.rows + FX_TY - 1) / FX_TY);
    A.lz = march_planes((long long)tiles * A.M, A.dir.planes, SMAX, fixed_per_sm(SMAX), 1.0, 0.9, A.M > 1, 65535 / A.M);
    A.nzb = (A.dir.planes + A.lz - 1) / A.lz;
    march_order(A, (long long)tiles * A.M * A.nzb, fixed_per_sm(SMAX));
    return launch_pdl(k_shell_fixed<SMAX>, dim3(tiles, 1, A.M * A.nzb), 64 * FX_TY, smem, st, maps, A);
}

}  // namespace lbe
