// K2: contact values (Appendix: g_ab evaluated at contact, a functional of the
// densities).  Per node:
//   n-bar_b = (1/|B_b|) sum_{|d| <= sigma_b/2} n_b(r + d)      (ball average)
//   xi_k    = (pi/6) sum_b sigma_b^k n-bar_b,  k = 2, 3
//   g_ab    = 1/(1-xi3) + 3 s xi2/(1-xi3)^2 + 2 s^2 xi2^2/(1-xi3)^3,
//             s = sigma_a sigma_b/(sigma_a + sigma_b)   (Boublik-Mansoori-
//             Carnahan-Starling-Leland contact value)
// Outputs: g_ab [M][M][N] and the padded fields the shell-force kernels stream, with their periodic
// images: g_ab n_b [M][M][P] in FP64; in FP32 the deviations n_b - ref_b [M][P] and g_ab n_b - ref_ab
// [M][M][P] from reference values (lbe_shell_march.cuh); optionally xi2 and xi3 [2][N] (kept for the
// discrete adjoint).
//
// MODE 1 is the transpose of the ball average for the discrete adjoint: the
// same march sums a padded field per species over the ball, and the kernel
// adds the sums to ln [M][N] (zero on solid nodes, whose density is fixed).
// The ball is symmetric, so its transpose is the same sum.
//
// Data path: the padded densities of all species are streamed plane by plane into a shared-memory ring by
// TMA; a block marches one tile along z.  The ball's section at height |dz| is a disc, and the discs are nested:
// one pass over the rows of the input plane (+dy and -dy combined, then summed outwards from dx = 0) yields the
// sums over all sections, which are added to the running sums of the outputs z - R .. z + R they belong to
// (registers, shifted by one per plane by the add's own destination).  A plane is read once.  FP32 threads own
// two outputs along x, packed as f32x2: 19 loads of 8 bytes for two outputs of the diameter-6 ball, where the
// sum over the ball's points read 123 values for one.  The halo's periodic images are written by their own node,
// one offset for all fields (an address per field and image doubled the time of the tiles at the edges).
// Contact stage on GB300, before (sum over the ball's points from a ring of 2R + 2 planes; spectral on the wells)
// and now: 512x128x128 channel of diameters 4 and 6 251 -> 96 us, 256^3 well of diameter 6 373 -> 122 us, 64^3
// well 50 -> 14 us, 90x75x66 with diameters 2, 4 and 6 129 -> 31 us, 1024x1024x1 of diameters 4 and 6 158 -> 103 us.
#pragma once
#include <algorithm>
#include <atomic>
#include <utility>

#include "lbe_device.cuh"
#include "lbe_launch.h"
#include "lbe_march.cuh"

namespace lbe {

constexpr int CT_THREADS = 128;

template <typename T, int M, int RB>
struct ContactTile {
    static constexpr int A = 16 / (int)sizeof(T);
    static constexpr int NX = sizeof(T) == 4 ? 2 : 1;  // outputs along x per thread
    static constexpr int TX = 32;
    static constexpr int TY = CT_THREADS * NX / TX;
    static constexpr int HX = (RB + A - 1) / A * A;  // halo along x: keeps the copies on 16-byte boundaries
    static constexpr int BX = TX + 2 * HX;
    static constexpr int BY = TY + 2 * RB;
    static constexpr int R = RB + 3;  // ring slots: the plane in use, RB behind it (centre values), two in flight
    static constexpr int PLANE = BX * BY;
    static constexpr int PLANE_BYTES = ((PLANE * (int)sizeof(T)) + 127) / 128 * 128;
    static constexpr int SLOT_BYTES = M * PLANE_BYTES;
    static constexpr int SMEM = R * SLOT_BYTES + 256 + 128;
};

// The values of a thread's outputs: packed FP32 pairs, or one FP64 value.  Row<E> holds a row of the plane
// around them, X = -E .. E; at an odd X a packed value consists of the halves of two loads.
template <typename T>
struct Lane;
template <>
struct Lane<float> {
    using V = f2;
    static __device__ __forceinline__ V zero() { return 0ull; }
    static __device__ __forceinline__ V add(V a, V b) { return f2add(a, b); }
    template <int E>
    struct Row {
        static constexpr int E2 = (E + 1) / 2 * 2;
        f2 v[E2 + 1];
        __device__ __forceinline__ void load(const float *c) {
#pragma unroll
            for (int i = 0; i <= E2; ++i) v[i] = *reinterpret_cast<const f2 *>(c - E2 + 2 * i);
        }
        template <int X>
        __device__ __forceinline__ float lo() const {
            return X % 2 == 0 ? f2unpack(v[(E2 + X) / 2]).x : f2unpack(v[(E2 + X - 1) / 2]).y;
        }
        template <int X>
        __device__ __forceinline__ float hi() const {
            return X % 2 == 0 ? f2unpack(v[(E2 + X) / 2]).y : f2unpack(v[(E2 + X + 1) / 2]).x;
        }
        // value at X of this row plus value at Y of row o (X and Y of the same parity)
        template <int X, int Y>
        __device__ __forceinline__ V sum(const Row &o) const {
            if constexpr (X % 2 == 0) return f2add(v[(E2 + X) / 2], o.v[(E2 + Y) / 2]);
            return f2pack(lo<X>() + o.template lo<Y>(), hi<X>() + o.template hi<Y>());
        }
        __device__ __forceinline__ V centre() const { return v[E2 / 2]; }
    };
};
template <>
struct Lane<double> {
    using V = double;
    static __device__ __forceinline__ V zero() { return 0.0; }
    static __device__ __forceinline__ V add(V a, V b) { return a + b; }
    template <int E>
    struct Row {
        double v[2 * E + 1];
        __device__ __forceinline__ void load(const double *c) {
#pragma unroll
            for (int i = 0; i <= 2 * E; ++i) v[i] = c[i - E];
        }
        template <int X, int Y>
        __device__ __forceinline__ V sum(const Row &o) const {
            return v[E + X] + o.v[E + Y];
        }
        __device__ __forceinline__ V centre() const { return v[E]; }
    };
};

// Balls |d| <= sigma/2 by their largest |d|^2.  An integer sigma has floor(sigma^2 / 4); the diameters accepted may lie
// a rounding below an even one (5.999999999999999 from a division), whose ball ends before the points at sigma/2:
// 3, 8 and 14 for 4, 6 and 8 (and 0 for 2).
constexpr int NBALLS = 12;
__host__ __device__ constexpr int ball_d2(int k) {
    constexpr int d2[NBALLS] = {0, 1, 2, 3, 4, 6, 8, 9, 12, 14, 16, 20};
    return d2[k];
}
__host__ __device__ constexpr int ball_radius(int d2) {  // floor of the root
    int r = 0;
    while ((r + 1) * (r + 1) <= d2) ++r;
    return r;
}

// Largest a with a^2 + dy^2 + Z^2 <= D2, or -1: half-width of row dy of the ball's section at height Z.
__host__ __device__ constexpr int ball_row(int d2, int dy, int Z) {
    int a = -1;
    while ((a + 1) * (a + 1) + dy * dy + Z * Z <= d2) ++a;
    return a;
}

// Sums of the plane around c over the sections of the ball |d|^2 <= D2: D[Z], Z = 0 .. its radius <= RB.
template <typename T, int BX, int D2, int RB>
__device__ __forceinline__ void ball_sections(const T *c, typename Lane<T>::V (&D)[RB + 1]) {
    using Ln = Lane<T>;
    using V = typename Ln::V;
    constexpr int R = ball_radius(D2);
    [&]<int... DY>(std::integer_sequence<int, DY...>) {
        (
            [&] {
                constexpr int dy = DY;
                constexpr int E = ball_row(D2, dy, 0);
                typename Ln::template Row<E> rp, rm;
                rp.load(c + dy * BX);
                if constexpr (dy > 0) rm.load(c - dy * BX);
                V s = dy == 0 ? rp.centre() : Ln::add(rp.centre(), rm.centre());
                [&]<int... A>(std::integer_sequence<int, A...>) {
                    (
                        [&] {
                            constexpr int a = A;
                            if constexpr (a > 0) {
                                if constexpr (dy == 0)
                                    s = Ln::add(s, rp.template sum<a, -a>(rp));
                                else
                                    s = Ln::add(s, Ln::add(rp.template sum<a, a>(rm), rp.template sum<-a, -a>(rm)));
                            }
                            [&]<int... Z>(std::integer_sequence<int, Z...>) {
                                (
                                    [&] {
                                        if constexpr (ball_row(D2, dy, Z) == a) D[Z] = dy == 0 ? s : Ln::add(D[Z], s);
                                    }(),
                                    ...);
                            }(std::make_integer_sequence<int, R + 1>{});
                        }(),
                        ...);
                }(std::make_integer_sequence<int, E + 1>{});
            }(),
            ...);
    }(std::make_integer_sequence<int, R + 1>{});
}

struct ContactMaps {
    CUtensorMap m[MAXS];
};
template <typename T>
struct ContactConst {
    int ball[MAXS];      // the species' balls (ball_d2)
    int lz;              // output planes per block
    T c2[MAXS], c3[MAXS];  // (pi/6) sigma^k over the points of the ball: the sums' weights in xi_k
    T s1[MAXS][MAXS], s2[MAXS][MAXS];  // 3 s_ab, 2 s_ab^2
    float refn[MAXS];    // FP32: reference values of the deviations
    float refg[MAXS][MAXS];
};

// Periodic images of a node along one axis: copies k0 .. k1 of it lie inside the padded field.
struct Images {
    int k0, k1;
};
__device__ __forceinline__ Images images(int v, int n, int H, int periodic) {
    Images im{0, 0};
    if (periodic && (v < H || v >= n - H)) {
        im.k0 = -((v + H) / n);
        im.k1 = (n + H - 1 - v) / n;
    }
    return im;
}

template <typename T, int M, int RB, int MODE>
__global__ void __launch_bounds__(CT_THREADS)
    k_contact_tma(const __grid_constant__ ContactMaps maps, Grid g, ContactConst<T> cs, T *__restrict__ gab,
                  T *__restrict__ npad2, T *__restrict__ gnpad, T *__restrict__ xi_out,
                  const uint32_t *__restrict__ mask, T *__restrict__ ln, unsigned *__restrict__ top, int *err) {
    using Tl = ContactTile<T, M, RB>;
    using Ln = Lane<T>;
    using V = typename Ln::V;
    constexpr int NX = Tl::NX;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *base = smem_align128(smem_raw);
    uint64_t *bars = reinterpret_cast<uint64_t *>(base + Tl::R * Tl::SLOT_BYTES);
    constexpr int PL = Tl::PLANE_BYTES / (int)sizeof(T);

    const int tid = threadIdx.x;
    const int tx = tid % (32 / NX) * NX, ty = tid / (32 / NX);
    const int nbx = (g.nx + Tl::TX - 1) / Tl::TX;  // tiles of a plane lie along the grid's x, which has room for all
    const int x0 = blockIdx.x % nbx * Tl::TX, y0 = blockIdx.x / nbx * Tl::TY, z0 = blockIdx.z * cs.lz;
    const int nout = min(cs.lz, g.nz - z0);
    const int nplanes = nout + 2 * RB;
    const bool leader = tid == 0;
    const int bx = x0 + g.H - Tl::HX;
    const int by = y0 + g.H - RB;
    constexpr uint32_t tx_bytes = (uint32_t)M * Tl::PLANE * (uint32_t)sizeof(T);

    if (leader) {
        for (int b = 0; b < M; ++b) prefetch_tensormap(&maps.m[b]);
        for (int r = 0; r < Tl::R; ++r) mbar_init(&bars[r], 1);
        fence_mbar_init();
    }
    __syncthreads();
    pdl_wait();
    auto issue = [&](int j) {
        const int slot = j % Tl::R;
        unsigned char *dst = base + slot * Tl::SLOT_BYTES;
        const int zp = z0 - RB + j + g.H;
        mbar_arrive_expect_tx(&bars[slot], tx_bytes);
#pragma unroll
        for (int b = 0; b < M; ++b) tma_load_3d(dst + b * Tl::PLANE_BYTES, &maps.m[b], bx, by, zp, &bars[slot]);
    };
    if (leader)
        for (int j = 0; j < Tl::R && j < nplanes; ++j) issue(j);

    const int x = x0 + tx, y = y0 + ty;
    const bool active = x < g.nx && y < g.ny, both = NX == 2 && active && x + 1 < g.nx;
    const bool vec = (g.nx & 1) == 0;  // rows of [N] fields start on 8-byte boundaries
    const int toff = (ty + RB) * Tl::BX + tx + Tl::HX;
    // images of the thread's outputs inside the halo of the padded fields
    const Images ix0 = images(x, g.nx, g.H, g.per[0]), ix1 = images(x + NX - 1, g.nx, g.H, g.per[0]);
    const Images iy = images(y, g.ny, g.H, g.per[1]);
    const bool edge = (ix0.k0 | ix0.k1 | ix1.k0 | ix1.k1 | iy.k0 | iy.k1) != 0;
    unsigned i = (unsigned)x + (unsigned)g.nx * ((unsigned)y + (unsigned)g.ny * (unsigned)z0);
    long long pc = pidx(g, x, y, z0);
    const long long pxy = (long long)g.px * g.py;

    V acc[M][2 * RB + 1];  // running ball sums of the outputs z_in - RB .. z_in + RB
#pragma unroll
    for (int b = 0; b < M; ++b)
#pragma unroll
        for (int k = 0; k <= 2 * RB; ++k) acc[b][k] = Ln::zero();

    // FP64: high words of the largest values this thread writes (they order like the values)
    constexpr int NT = sizeof(T) == 8 && MODE == 0 ? M + M * M : 1;
    unsigned big[NT];
#pragma unroll
    for (int f = 0; f < NT; ++f) big[f] = 0;

    int slot = 0, cslot = Tl::R - RB;  // ring slots of the input plane and of the plane RB behind it
    if (cslot == Tl::R) cslot = 0;
    uint32_t ph = 0;
    for (int j = 0; j < nplanes; ++j) {
        if (!mbar_wait_bounded(&bars[slot], ph, err)) {
            mbar_drain(bars, Tl::R, j, min(max(Tl::R, j + Tl::R - RB), nplanes));
            return;
        }
        const T *sp = reinterpret_cast<const T *>(base + slot * Tl::SLOT_BYTES) + toff;
#pragma unroll
        for (int b = 0; b < M; ++b) {
            V D[RB + 1];
#pragma unroll
            for (int Z = 0; Z <= RB; ++Z) D[Z] = Ln::zero();
            const T *c = sp + b * PL;
            const int ball = cs.ball[b];
            [&]<int... K>(std::integer_sequence<int, K...>) {
                (
                    [&] {
                        constexpr int k = NBALLS - 1 - K, r = ball_radius(ball_d2(k));
                        // one species: a ball of the launch's radius
                        if constexpr (r == RB || (M > 1 && r < RB))
                            if (ball == k) ball_sections<T, Tl::BX, ball_d2(k), RB>(c, D);
                    }(),
                    ...);
            }(std::make_integer_sequence<int, NBALLS>{});
            // shift the running sums by one plane and add this plane's sections: output RB +- Z
#pragma unroll
            for (int k = 0; k < 2 * RB; ++k) acc[b][k] = Ln::add(acc[b][k + 1], D[k < RB ? RB - k : k - RB]);
            acc[b][2 * RB] = D[RB];
        }
        if (j >= 2 * RB) {
            // acc[.][0]: the output RB planes behind the input plane
            const int z = z0 + j - 2 * RB;
            if (active) {
                if constexpr (MODE == 1) {
                    // transpose of the ball average: add the ball sums of the species' fields to ln
#pragma unroll
                    for (int o = 0; o < NX; ++o) {
                        if (o == 1 && !both) continue;
                        const bool solid = mask[i + o] & 1u;
#pragma unroll
                        for (int b = 0; b < M; ++b) {
                            T *p = ln + (long long)b * g.N + i + o;
                            T v;
                            if constexpr (NX == 2)
                                v = o ? f2unpack(acc[b][0]).y : f2unpack(acc[b][0]).x;
                            else
                                v = acc[b][0];
                            *p = solid ? (T)0 : *p + v;
                        }
                    }
                } else {
                    const T *sc = reinterpret_cast<const T *>(base + cslot * Tl::SLOT_BYTES) + toff;
                    T nloc[M][NX], xi2[NX], xi3[NX], t2[NX], t3[NX], i1[NX];
                    bool bad = false;
#pragma unroll
                    for (int o = 0; o < NX; ++o) xi2[o] = xi3[o] = 0;
#pragma unroll
                    for (int b = 0; b < M; ++b) {
                        T s[NX];
                        if constexpr (NX == 2) {
                            const float2 u = f2unpack(acc[b][0]);
                            const float2 n2 = *reinterpret_cast<const float2 *>(sc + b * PL);
                            s[0] = u.x;
                            s[NX - 1] = u.y;
                            nloc[b][0] = n2.x;
                            nloc[b][NX - 1] = n2.y;
                        } else {
                            s[0] = acc[b][0];
                            nloc[b][0] = sc[b * PL];
                        }
#pragma unroll
                        for (int o = 0; o < NX; ++o) {
                            xi2[o] += cs.c2[b] * s[o];
                            xi3[o] += cs.c3[b] * s[o];
                        }
                    }
#pragma unroll
                    for (int o = 0; o < NX; ++o) {
                        i1[o] = (T)1 / ((T)1 - xi3[o]);
                        t2[o] = xi2[o] * i1[o] * i1[o];
                        t3[o] = xi2[o] * t2[o] * i1[o];
                        bad = bad || ((o == 0 || both) && !(xi3[o] < (T)1));
                        if (xi_out && (o == 0 || both)) {
                            xi_out[i + o] = xi2[o];
                            xi_out[g.N + i + o] = xi3[o];
                        }
                    }
                    // the padded outputs: FP32 n_b - ref_b, then g_ab n_b (- ref_ab) of every ordered pair
                    constexpr int ND = sizeof(T) == 4 ? M : 0;
                    T pv[ND + M * M][NX];
                    if constexpr (ND > 0) {
#pragma unroll
                        for (int b = 0; b < M; ++b)
#pragma unroll
                            for (int o = 0; o < NX; ++o) pv[b][o] = nloc[b][o] - cs.refn[b];
                    }
#pragma unroll
                    for (int a = 0; a < M; ++a)
#pragma unroll
                        for (int b = a; b < M; ++b) {
                            // s_ab and so g_ab are the same for (a, b) and (b, a)
                            T gv[NX];
#pragma unroll
                            for (int o = 0; o < NX; ++o) {
                                gv[o] = i1[o] + cs.s1[a][b] * t2[o] + cs.s2[a][b] * t3[o];
                                bad = bad || ((o == 0 || both) && !isfinite(gv[o]));
                            }
#pragma unroll
                            for (int h = 0; h < (a == b ? 1 : 2); ++h) {
                                const int a2 = h ? b : a, b2 = h ? a : b;
                                T *q = gab + (long long)(a2 * M + b2) * g.N + i;
                                if constexpr (NX == 2) {
                                    store_pair(q, f2pack(gv[0], gv[NX - 1]), vec, both);
#pragma unroll
                                    for (int o = 0; o < NX; ++o)
                                        pv[ND + a2 * M + b2][o] = fmaf(gv[o], nloc[b2][o], -cs.refg[a2][b2]);
                                } else {
                                    *q = gv[0];
                                    pv[a2 * M + b2][0] = gv[0] * nloc[b2][0];
                                }
                            }
                        }
                    if constexpr (sizeof(T) == 8) {
#pragma unroll
                        for (int b = 0; b < M; ++b)
                            big[b] = max(big[b], (unsigned)__double2hiint(nloc[b][0]) & 0x7fffffffu);
#pragma unroll
                        for (int f = 0; f < M * M; ++f)
                            big[M + f] = max(big[M + f], (unsigned)__double2hiint(pv[f][0]) & 0x7fffffffu);
                    }
                    auto field = [&](int f) -> T * {
                        return f < ND ? npad2 + (long long)f * g.P : gnpad + (long long)(f - ND) * g.P;
                    };
#pragma unroll
                    for (int f = 0; f < ND + M * M; ++f) {
                        T *q = field(f) + pc;
                        if constexpr (NX == 2) {  // x + H is even, rows hold a multiple of 8 elements
                            if (both)
                                *reinterpret_cast<float2 *>(q) = make_float2(pv[f][0], pv[f][NX - 1]);
                            else
                                q[0] = pv[f][0];
                        } else {
                            q[0] = pv[f][0];
                        }
                    }
                    // the periodic images inside the halo: one offset for all fields; along y and z a pair stays one
                    // store (two stores of every other value: 310 instead of 103 us on 1024x1024x1, two species)
                    const Images iz = images(z, g.nz, g.H, g.per[2]);
                    if (edge || (iz.k0 | iz.k1) != 0) {
                        for (int kz = iz.k0; kz <= iz.k1; ++kz)
                            for (int ky = iy.k0; ky <= iy.k1; ++ky) {
                                const long long d =
                                    pc + (long long)g.px * (ky * g.ny + (long long)g.py * (kz * g.nz));
                                if ((ky | kz) != 0) {
#pragma unroll
                                    for (int f = 0; f < ND + M * M; ++f) {
                                        T *q = field(f) + d;
                                        if (NX == 2 && both)
                                            *reinterpret_cast<float2 *>(q) = make_float2(pv[f][0], pv[f][NX - 1]);
                                        else
                                            q[0] = pv[f][0];
                                    }
                                }
#pragma unroll
                                for (int o = 0; o < NX; ++o) {
                                    if (o == 1 && !both) continue;
                                    const Images ix = o ? ix1 : ix0;
                                    for (int kx = ix.k0; kx <= ix.k1; ++kx) {
                                        if (kx == 0) continue;
#pragma unroll
                                        for (int f = 0; f < ND + M * M; ++f) field(f)[d + o + kx * g.nx] = pv[f][o];
                                    }
                                }
                            }
                    }
                    if (bad) atomicOr(err, ERR_PACKING);
                }
            }
            i += (unsigned)(g.nx * g.ny);
            pc += pxy;
        }
        __syncthreads();
        // the plane RB behind was read for the last time: its slot takes the next copy
        if (leader && j >= RB && j + Tl::R - RB < nplanes) {
            fence_proxy_async_smem();
            issue(j + Tl::R - RB);
        }
        if (++slot == Tl::R) {
            slot = 0;
            ph ^= 1u;
        }
        if (++cslot == Tl::R) cslot = 0;
    }
    if constexpr (sizeof(T) == 8 && MODE == 0) {
#pragma unroll
        for (int f = 0; f < NT; ++f) {
            const unsigned m = __reduce_max_sync(0xffffffffu, big[f]);
            // most warps find the maximum raised already
            if ((tid & 31) == 0 && m > *(volatile unsigned *)(top + f)) atomicMax(top + f, m);
        }
    }
}

template <typename T, int M, int RB, int MODE>
cudaError_t launch_ct(const ContactLaunch &L, cudaStream_t st) {
    using Tl = ContactTile<T, M, RB>;
    static PerDevice once;
    cudaError_t e = allow_smem(once, k_contact_tma<T, M, RB, MODE>, Tl::SMEM);
    if (e != cudaSuccess) return e;
    static std::atomic<int> resident{0};  // blocks per SM, the same on every device this library runs on
    int per_sm = resident.load(std::memory_order_relaxed);
    if (per_sm == 0) {
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_contact_tma<T, M, RB, MODE>, CT_THREADS, Tl::SMEM);
        if (e != cudaSuccess) return e;
        per_sm = per_sm > 0 ? per_sm : 1;
        resident.store(per_sm, std::memory_order_relaxed);
    }
    const Grid &g = *L.grid;
    ContactMaps maps;
    for (int b = 0; b < M; ++b) maps.m[b] = L.maps[b];
    ContactConst<T> cs{};
    for (int b = 0; b < M; ++b) {
        int d2 = 0;  // of the rows that also normalise the average
        for (int dz = -4; dz <= 4; ++dz)
            for (int k = L.br->first[b][dz + 4]; k < L.br->first[b][dz + 5]; ++k)
                d2 = std::max(d2, dz * dz + L.br->dy[b][k] * L.br->dy[b][k] + L.br->a[b][k] * L.br->a[b][k]);
        cs.ball[b] = -1;
        for (int k = 0; k < NBALLS; ++k)
            if (ball_d2(k) == d2) cs.ball[b] = k;
        if (cs.ball[b] < 0) return cudaErrorInvalidValue;
        cs.c2[b] = (T)(L.cp->xi2c[b] / L.br->count[b]);
        cs.c3[b] = (T)(L.cp->xi3c[b] / L.br->count[b]);
        cs.refn[b] = (float)L.refn[b];
        for (int a = 0; a < M; ++a) {
            const double s = L.cp->s_ab[a][b];
            cs.refg[a][b] = (float)L.refg[a][b];
            cs.s1[a][b] = (T)(3.0 * s);
            cs.s2[a][b] = (T)(2.0 * s * s);
        }
    }
    const int tiles = (g.nx + Tl::TX - 1) / Tl::TX * ((g.ny + Tl::TY - 1) / Tl::TY);
    cs.lz = march_planes(tiles, g.nz, RB, per_sm, 0.35, 2.4, false, 65535);
    dim3 grid(tiles, 1, (g.nz + cs.lz - 1) / cs.lz);
    return launch_pdl(k_contact_tma<T, M, RB, MODE>, grid, CT_THREADS, Tl::SMEM, st, maps, g, cs, (T *)L.gab,
                      (T *)L.npad2, (T *)L.gnpad, (T *)L.xi, L.mask, (T *)L.ln, L.top, L.err);
}

template <typename T, int M, int MODE>
cudaError_t dispatch_rb(const ContactLaunch &L, cudaStream_t st) {
    switch (L.RB) {
        case 0: return launch_ct<T, M, 0, MODE>(L, st);
        case 1: return launch_ct<T, M, 1, MODE>(L, st);
        case 2: return launch_ct<T, M, 2, MODE>(L, st);
        case 3: return launch_ct<T, M, 3, MODE>(L, st);
        case 4: return launch_ct<T, M, 4, MODE>(L, st);
        default: return cudaErrorInvalidValue;
    }
}

template <typename T, int MODE>
cudaError_t dispatch_m(const ContactLaunch &L, cudaStream_t st) {
    switch (L.cp->M) {
        case 1: return dispatch_rb<T, 1, MODE>(L, st);
        case 2: return dispatch_rb<T, 2, MODE>(L, st);
        case 3: return dispatch_rb<T, 3, MODE>(L, st);
        case 4: return dispatch_rb<T, 4, MODE>(L, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace lbe
