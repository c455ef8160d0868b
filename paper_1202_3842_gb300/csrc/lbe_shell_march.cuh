// K3 in FP32: mean-field Enskog force (Appendix, hard-sphere C^{alpha,mf})
//   C^a(r) = sum_b coef_ab n_a(r) [ g_ab(r)/2 P_ab(r) + Q_ab(r)/2 ],
//   P_ab = sum_{e in K_ab} e^ n_b(r+e),  Q_ab = sum_{e in K_ab} e^ (g_ab n_b)(r+e),
// coef_ab = -kT sigma_ab^2 w_ab, for every pair of every species in one launch.
//
// A shell sum of an odd kernel is the same for every constant added to its field, so the fields are
// kept as deviations from a reference value (the padded fields hold -ref on solid nodes and beyond
// closed axes, where the density is 0): sums of like values then round relative to the deviations.
//
// Scatter along z.  A block marches one tile through z and reads each input plane once.  Of a plane,
// the points (+-X, +-Y) of the shell's projection are combined once,
//   x: a - b + c - d,  y: a + b - c - d,  z: a + b + c + d   (a..d the four corners),
// weighted for every |Z| at which (X, Y, Z) lies in the shell, and summed into B_x, B_y, B_z (|Z|).
// The plane's B(|Z|) are then added to the running sums of the 2S + 1 outputs z_in - S .. z_in + S, which
// a thread keeps in registers and shifts by one per plane (the shift is the add's own destination).  At
// S = 6 that takes about 440 operations per output and field where the sum over the half shell, point by
// point, takes 731, and a plane's values are read once instead of once for each z-block.  The plane in
// use is all that shared memory has to hold (the gather needs 2S + 1 planes), so three blocks share an
// SM, and the loop body is a fourth of the unrolled half shell's code.
//
// Bound by the FP32 pipe.  Two outputs along x per thread, packed as f32x2: a row of the projection is
// then read by aligned 8-byte loads that serve both outputs (79 loads for two outputs of one field at
// S = 6), and odd X take their operands from the halves of two loads (scalar adds, same pipe time).
// The two fields of a pair run in separate warps of a block; P reaches the warps that finish C through
// shared memory.  What C's epilogue reads from global memory is loaded one plane ahead (read in the plane's
// own pass, its latency showed: 1190 instead of 1010 us on the 512x128x128 channel).
//
// The march goes along z with tiles of 32 x 4 nodes in x and y, or along y with tiles in x and z where few nodes lie
// along z (march_axes): each cut of a march reads 2S planes again.
//
// Shell stage on GB300, against the half-shell stencils it replaces (y-blocked for diameters 4 to 6, z-blocked
// else; spectral on the wells): 512x128x128 channel of diameters 4 and 6 1566 -> 996 us, 256^3 well of diameter
// 6 776 -> 638 us, 64^3 well 50 -> 35 us, 128x32x32 channel 184 -> 45 us, 90x75x66 with diameters 2, 4 and 6
// 311 -> 163 us, 1024x1024x1 of diameter 6 220 -> 177 us, of diameter 8 250 -> 289 us.  The channel's operations
// (439 per output and field at diameter 6, without the halo planes) take the FP32 pipe 55% of that time.  On the 160^3 well the pipe is busy 64% of the active cycles at 2.2 warps per scheduler
// (162 registers); the rest is dependent issue ("wait" 0.9 cycles per instruction).
//
// Error of C in FP32 against FP64, rms over the root of the sum of squares on the shell (half-shell stencils in
// brackets): 1% noise, diameter 6, 3.5e-8 (8.1e-8); density over one decade along x 4.8e-7 1.2e-7 2.3e-7 in x, y, z
// (6.1e-7 1.4e-7 1.4e-7), over three, where it is 1e-3 to 1e-2 of its largest, 4.1e-5 6.9e-7 2.0e-6 (4.1e-5 6.9e-7
// 6.6e-7: there the densities themselves, stored as deviations from n0, are off by 6e-5).  z sums like values that
// cancel between planes.
#pragma once
#include "lbe_launch.h"
#include "lbe_march.cuh"

namespace lbe {

constexpr int SM_TY = 4;  // output rows of a tile (32 x SM_TY outputs per plane)
constexpr int SM_R = 4;  // ring slots

template <int S>
struct ShellMarchTile {
    static constexpr int S4 = (S + 3) / 4 * 4;  // halo along x: keeps the copies on 16-byte boundaries
    static constexpr int BX = 32 + 2 * S4;
    static constexpr int BY = SM_TY + 2 * S;
    static constexpr int PLANE = BX * BY;
    static constexpr int PLANE_BYTES = (PLANE * 4 + 127) / 128 * 128;
    static constexpr int SLOT_BYTES = 2 * PLANE_BYTES;
};
// Blocks per SM: a thread's registers hold 6 SMAX running sums (packed pairs) besides the plane's B.
__host__ __device__ constexpr int shell_march_per_sm(int smax) {
    return (smax <= 4 ? 16 : (smax <= 6 ? 12 : 8)) / SM_TY;
}
template <int SMAX>
struct ShellMarchSmem {
    static constexpr int SLOT = ShellMarchTile<SMAX>::SLOT_BYTES;
    static constexpr int XCH = SM_R * SLOT;  // P exchange: [2][3][16 SM_TY] f2
    static constexpr int BARS = XCH + 2 * 3 * 16 * SM_TY * 8;
    static constexpr int BYTES = BARS + SM_R * 8 + 128;
};

// Whether (X, Y) is the first point, in the order the plane is walked, that adds to component c of B(Z).
__host__ __device__ constexpr bool ring_first(int S, int X, int Y, int Z, int c) {
    for (int y = 0; y <= Y; ++y)
        for (int x = 0; x <= S && (y < Y || x < X); ++x)
            if (in_shell(S, x, y, Z) && (c == 2 || (c == 0 ? x > 0 : y > 0))) return false;
    return true;
}
template <bool FIRST>
__device__ __forceinline__ void march_add(f2 &B, float w, f2 v) {
    B = FIRST ? f2mul(f2splat(w), v) : f2fma(f2splat(w), v, B);
}

// One row pair (Y, -Y) of the plane's projection; c points at the thread's first output.
template <int S, int Y>
__device__ __forceinline__ void march_rows(const float *c, f2 *Bx, f2 *By, f2 *Bz) {
    constexpr int BX = ShellMarchTile<S>::BX;
    constexpr int E = (ring_xmax(S, Y) + 1) / 2 * 2;
    f2 rp[E + 1], rm[E + 1] = {};  // the rows' values at X = -E, -E + 2, .. E (and the next one of each)
#pragma unroll
    for (int i = 0; i <= E; ++i) {
        rp[i] = *reinterpret_cast<const f2 *>(c + Y * BX - E + 2 * i);
        if constexpr (Y > 0) rm[i] = *reinterpret_cast<const f2 *>(c - Y * BX - E + 2 * i);
    }
    [&]<int... XI>(std::integer_sequence<int, XI...>) {
        (
            [&] {
                constexpr int X = XI;
                constexpr unsigned m = ring_mask(S, X, Y);
                if constexpr (m != 0) {
                    f2 dx = 0, dy = 0, sz = 0;
                    if constexpr (X == 0 && Y == 0) {
                        sz = rp[E / 2];
                    } else if constexpr (X == 0) {
                        dy = f2sub(rp[E / 2], rm[E / 2]);
                        sz = f2add(rp[E / 2], rm[E / 2]);
                    } else if constexpr (X % 2 == 0) {
                        const f2 a = rp[(E + X) / 2], b = rp[(E - X) / 2];
                        if constexpr (Y == 0) {
                            dx = f2sub(a, b);
                            sz = f2add(a, b);
                        } else {
                            const f2 cc = rm[(E + X) / 2], d = rm[(E - X) / 2];
                            const f2 u = f2sub(a, d), v = f2sub(cc, b);
                            dx = f2add(u, v);
                            dy = f2sub(u, v);
                            sz = f2add(f2add(a, d), f2add(b, cc));
                        }
                    } else {
                        // odd X: the outputs' values are the halves of two neighbouring loads
                        const float a0 = f2unpack(rp[(E + X - 1) / 2]).y, a1 = f2unpack(rp[(E + X + 1) / 2]).x;
                        const float b0 = f2unpack(rp[(E - X - 1) / 2]).y, b1 = f2unpack(rp[(E - X + 1) / 2]).x;
                        if constexpr (Y == 0) {
                            dx = f2pack(a0 - b0, a1 - b1);
                            sz = f2pack(a0 + b0, a1 + b1);
                        } else {
                            const float c0 = f2unpack(rm[(E + X - 1) / 2]).y, c1 = f2unpack(rm[(E + X + 1) / 2]).x;
                            const float d0 = f2unpack(rm[(E - X - 1) / 2]).y, d1 = f2unpack(rm[(E - X + 1) / 2]).x;
                            const f2 u = f2pack(a0 - d0, a1 - d1), v = f2pack(c0 - b0, c1 - b1);
                            dx = f2add(u, v);
                            dy = f2sub(u, v);
                            sz = f2add(f2pack(a0 + d0, a1 + d1), f2pack(b0 + c0, b1 + c1));
                        }
                    }
                    [&]<int... ZI>(std::integer_sequence<int, ZI...>) {
                        (
                            [&] {
                                constexpr int Z = ZI;
                                if constexpr ((m >> Z) & 1u) {
                                    constexpr double len = ct_sqrt((double)(X * X + Y * Y + Z * Z));
                                    if constexpr (X > 0)
                                        march_add<ring_first(S, X, Y, Z, 0)>(Bx[Z], (float)(X / len), dx);
                                    if constexpr (Y > 0)
                                        march_add<ring_first(S, X, Y, Z, 1)>(By[Z], (float)(Y / len), dy);
                                    if constexpr (Z > 0)
                                        march_add<ring_first(S, X, Y, Z, 2)>(Bz[Z], (float)(Z / len), sz);
                                }
                            }(),
                            ...);
                    }(std::make_integer_sequence<int, S + 1>{});
                }
            }(),
            ...);
    }(std::make_integer_sequence<int, ring_xmax(S, Y) + 1>{});
}

template <int S, int... Y>
__device__ __forceinline__ void march_plane(const float *c, f2 *Bx, f2 *By, f2 *Bz,
                                            std::integer_sequence<int, Y...>) {
    (march_rows<S, Y>(c, Bx, By, Bz), ...);
}

struct ShellMarchArgs {
    Grid g;
    MarchAxes dir;
    int M, lz, nzb;              // planes per block, blocks along z
    int order[MAXS];             // species in the order their blocks start
    int S[MAXS * MAXS];          // pair diameter of [a][b], 0: no pair
    int q[MAXS * MAXS];          // index of the pair in Pout
    float coef[MAXS * MAXS];
    const float *npad;           // densities [M][P]
    const float *gab;            // contact values [M][M][N]
    float *C;                    // [M][3][N]
    float *Pout;                 // NULL, or [pairs][3][N]
    int *err;
};
// March of one pair through the block's planes; `it` counts the planes of the block's ring.
template <int SMAX, int S>
__device__ __forceinline__ bool shell_march(const ShellMarchMaps &maps, const ShellMarchArgs &A, unsigned char *base,
                                            uint64_t *bars, int a, int b, int z0, int nout, bool accumulate, int &it) {
    using Tl = ShellMarchTile<S>;
    using Sm = ShellMarchSmem<SMAX>;
    const Grid &g = A.g;
    const MarchAxes &dir = A.dir;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int fld = warp / (SM_TY / 2);  // 0: P (n_b), 1: Q (g_ab n_b)
    const int ot = tid - fld * (16 * SM_TY);
    const int row = 2 * (warp - fld * (SM_TY / 2)) + (lane >> 4);
    const int tx = 2 * (lane & 15);
    const int nbx = (g.nx + 31) / 32;  // tiles of a plane lie along the grid's x, which has room for all
    const int x0 = blockIdx.x % nbx * 32, y0 = blockIdx.x / nbx * SM_TY;
    const int x = x0 + tx, y = y0 + row;
    const int pair = a * A.M + b;
    const int nplanes = nout + 2 * S;
    const bool leader = tid == 0;
    const int first_it = it;
    f2 *xch = reinterpret_cast<f2 *>(base + Sm::XCH);

    auto issue = [&](int j) {  // plane j holds interior z = z0 - S + j (z: along the march, y: along the rows)
        const int k = first_it + j, slot = k % SM_R;
        unsigned char *dst = base + slot * Sm::SLOT;
        const int bx = x0 + g.H - Tl::S4, by = y0 + g.H - S, zp = z0 - S + j + g.H;
        mbar_arrive_expect_tx(&bars[slot], 2u * Tl::PLANE * 4u);
        tma_load_3d(dst, &maps.n[pair], bx, dir.swap ? zp : by, dir.swap ? by : zp, &bars[slot]);
        tma_load_3d(dst + Tl::PLANE_BYTES, &maps.gn[pair], bx, dir.swap ? zp : by, dir.swap ? by : zp, &bars[slot]);
    };
    if (leader) {
        if (first_it > 0) fence_proxy_async_smem();  // the ring was read for the pair before
        for (int j = 0; j < SM_R && j < nplanes; ++j) issue(j);
    }

    f2 ax[2 * S], ay[2 * S], az[2 * S];
#pragma unroll
    for (int k = 0; k < 2 * S; ++k) ax[k] = ay[k] = az[k] = 0ull;
    const bool act0 = x < g.nx && y < dir.rows, act1 = act0 && x + 1 < g.nx;
    const bool vec = (g.nx & 1) == 0;  // rows start on 8-byte boundaries
    // node index of the output at hand (lattices hold fewer than 2^31 nodes); one 32-bit offset per thread from
    // the pair's base pointers, which are the same for the whole block
    unsigned i = (unsigned)x + dir.srow * (unsigned)y + dir.splane * (unsigned)z0;
    const f2 half_coef = f2splat(0.5f * A.coef[pair]);
    const int coff = (row + S) * Tl::BX + tx + Tl::S4;
    float *const Ca = A.C + 3 * (long long)a * g.N, *const Pa = A.Pout ? A.Pout + 3 * (long long)A.q[pair] * g.N : nullptr;
    const long long comp[3] = {0, march_component(g, dir, 1), march_component(g, dir, 2)};
    const float *gb = A.gab + (long long)pair * g.N;
    const float *np = A.npad + (long long)a * g.P + march_pidx(g, dir, x, y, z0);

    // what the epilogue reads from global memory, loaded one plane ahead; rows of the padded field start on
    // 8-byte boundaries and x is even, so its two outputs are one load (within the row)
    f2 na = 0, gr = 0, old[3] = {0, 0, 0};
    auto load_epilogue = [&] {
        na = *reinterpret_cast<const f2 *>(np);
        if (fld == 0) {
            gr = load_pair(gb + i, vec, act1);
        } else if (accumulate) {
#pragma unroll
            for (int c = 0; c < 3; ++c) old[c] = load_pair(Ca + comp[c] + i, vec, act1);
        }
    };
    if (act0) load_epilogue();

    for (int j = 0; j < nplanes; ++j) {
        const int k = first_it + j, slot = k % SM_R;
        if (!mbar_wait_bounded(&bars[slot], (uint32_t)(k / SM_R) & 1u, A.err)) {
            mbar_drain(bars, SM_R, k, first_it + min(j + SM_R, nplanes));
            return false;
        }
        const bool out = j >= 2 * S && act0;
        f2 Bx[S + 1], By[S + 1], Bz[S + 1];
        const float *c = reinterpret_cast<const float *>(base + slot * Sm::SLOT + fld * Tl::PLANE_BYTES) + coff;
        march_plane<S>(c, Bx, By, Bz, std::make_integer_sequence<int, S + 1>{});
        // output k of the march is S - k planes below the input plane: B(|S - k|), the z component odd
        f2 v[3] = {f2add(ax[0], Bx[S]), f2add(ay[0], By[S]), f2add(az[0], Bz[S])};
#pragma unroll
        for (int o = 1; o < 2 * S; ++o) {
            const int Z = o < S ? S - o : o - S;
            ax[o - 1] = f2add(ax[o], Bx[Z]);
            ay[o - 1] = f2add(ay[o], By[Z]);
            az[o - 1] = o == S ? az[o] : (o < S ? f2add(az[o], Bz[Z]) : f2sub(az[o], Bz[Z]));
        }
        ax[2 * S - 1] = Bx[S];
        ay[2 * S - 1] = By[S];
        az[2 * S - 1] = f2sub(0ull, Bz[S]);
        f2 *xo = xch + (j & 1) * (3 * 16 * SM_TY) + ot;
        const f2 pre = f2mul(na, half_coef);
        if (fld == 0 && out) {
            const f2 gp = f2mul(pre, gr);
#pragma unroll
            for (int cc = 0; cc < 3; ++cc) {
                xo[cc * (16 * SM_TY)] = f2mul(gp, v[cc]);
                if (Pa) store_pair(Pa + comp[cc] + i, v[cc], vec, act1);
            }
        }
        __syncthreads();
        if (leader && j + SM_R < nplanes) {
            fence_proxy_async_smem();
            issue(j + SM_R);
        }
        if (fld == 1 && out) {
#pragma unroll
            for (int cc = 0; cc < 3; ++cc)
                store_pair(Ca + comp[cc] + i, f2add(old[cc], f2fma(pre, v[cc], xo[cc * (16 * SM_TY)])), vec, act1);
        }
        if (j >= 2 * S) {
            i += dir.splane;
            np += dir.pplane;
            if (act0 && j + 1 < nplanes) load_epilogue();
        }
    }
    it = first_it + nplanes;
    return true;
}

template <int SMAX>
__global__ void __launch_bounds__(32 * SM_TY, shell_march_per_sm(SMAX))
    k_shell_march(const __grid_constant__ ShellMarchMaps maps, const __grid_constant__ ShellMarchArgs A) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char *base = smem_align128(smem_raw);
    uint64_t *bars = reinterpret_cast<uint64_t *>(base + ShellMarchSmem<SMAX>::BARS);
    const int k = blockIdx.z / A.nzb, a = A.order[k];
    const int z0 = (blockIdx.z - k * A.nzb) * A.lz;
    const int nout = min(A.lz, A.dir.planes - z0);
    if (threadIdx.x == 0) {
        for (int r = 0; r < SM_R; ++r) mbar_init(&bars[r], 1);
        fence_mbar_init();
    }
    __syncthreads();
    pdl_wait();
    if (nout <= 0) return;
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
                        ok = shell_march<SMAX, I + 1>(maps, A, base, bars, a, b, z0, nout, accumulate, it);
                }(),
                ...);
        }(std::make_integer_sequence<int, SMAX>{});
        if (!ok) return;
        accumulate = true;
    }
}

template <int SMAX>
cudaError_t launch_shell_march_t(const ShellMarchMaps &maps, ShellMarchArgs &A, cudaStream_t st) {
    constexpr int smem = ShellMarchSmem<SMAX>::BYTES;
    static PerDevice once;
    const cudaError_t e = allow_smem(once, k_shell_march<SMAX>, smem);
    if (e != cudaSuccess) return e;
    const Grid &g = A.g;
    const int tiles = (g.nx + 31) / 32 * ((A.dir.rows + SM_TY - 1) / SM_TY);
    constexpr int per_sm = shell_march_per_sm(SMAX);
    A.lz = march_planes((long long)tiles * A.M, A.dir.planes, SMAX, per_sm, 1.0, 0.9, A.M > 1, 65535 / A.M);
    A.nzb = (A.dir.planes + A.lz - 1) / A.lz;
    march_order(A, (long long)tiles * A.M * A.nzb, per_sm);
    return launch_pdl(k_shell_march<SMAX>, dim3(tiles, 1, A.M * A.nzb), 32 * SM_TY, smem, st, maps, A);
}

}  // namespace lbe
