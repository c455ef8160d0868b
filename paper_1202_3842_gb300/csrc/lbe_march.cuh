// Pieces shared by the kernels that march a tile through z and scatter each input plane into the
// outputs it reaches (the shell force K3 and the contact values K2): the plane rings of a shell, packed
// FP32 pairs, and the choice of the planes per block.
#pragma once
#include <utility>

#include "lbe_device.cuh"
#include "lbe_shell.cuh"

namespace lbe {

// Bit Z (0 <= Z <= S) is set when (X, Y, +-Z) lies in the shell of diameter S.
__host__ __device__ constexpr unsigned ring_mask(int S, int X, int Y) {
    unsigned m = 0;
    for (int z = 0; z <= S; ++z)
        if (in_shell(S, X, Y, z)) m |= 1u << z;
    return m;
}
// Largest |X| of a row Y of the shell's projection onto a plane (0 <= Y <= S; every row has some).
__host__ __device__ constexpr int ring_xmax(int S, int Y) {
    int r = 0;
    for (int x = 0; x <= S; ++x)
        if (ring_mask(S, x, Y)) r = x;
    return r;
}

// Packed pairs of FP32 values (x in the low half); each lane rounds like the scalar instruction.
using f2 = unsigned long long;
__device__ __forceinline__ f2 f2sub(f2 a, f2 b) {
    f2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 f2add(f2 a, f2 b) {
    f2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 f2mul(f2 a, f2 b) {
    f2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f2 f2fma(f2 a, f2 b, f2 c) {
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f2 f2pack(float x, float y) {
    f2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
    return d;
}
__device__ __forceinline__ f2 f2splat(float u) { return f2pack(u, u); }
__device__ __forceinline__ float2 f2unpack(f2 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}

__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// Two neighbouring values of a field: one 8-byte access where rows have an even length, else one by one (the
// second only inside the row).
__device__ __forceinline__ f2 load_pair(const float *p, bool vec, bool both) {
    if (vec) return *reinterpret_cast<const f2 *>(p);
    return f2pack(p[0], both ? p[1] : 0.f);
}
__device__ __forceinline__ void store_pair(float *p, f2 v, bool vec, bool both) {
    if (vec) {
        *reinterpret_cast<f2 *>(p) = v;
    } else {
        const float2 r = f2unpack(v);
        p[0] = r.x;
        if (both) p[1] = r.y;
    }
}

// Output planes per block of a marching kernel.  A block of lz outputs also reads 2 r halo planes, each at
// `halo` of an output plane's cost.  With b blocks per SM the chip takes per plane the time of b blocks,
// rounded up while all are resident (per_sm), plus `lat` blocks' worth of latency that too few blocks leave
// exposed; a partial last wave adds 0.4.  Short marches re-read the halo, long ones leave multiprocessors
// idle: the smallest product over all lz is taken (the longest march among equals).  The form and the
// constants of both kernels are fits to sweeps of lz on GB300 (512x128x128, 256^3, 128x32x32 and 64^3; within
// 10% of the measured times).
// Where blocks differ in length (`mixed`), a round of resident blocks takes less than its longest.
// At most `most` parts (a grid has 65535 blocks along z).
// `cost`: the product itself, in planes of one block per SM.
inline int march_planes(long long tiles, int nz, int r, int per_sm, double halo, double lat, bool mixed, int most,
                        double *cost_out = nullptr) {
    int best = 0;
    double cost = 0.0;
    for (int lz = (nz + most - 1) / most;;) {  // the shortest march of every number of parts
        const int parts = (nz + lz - 1) / lz;
        const double b = (double)tiles * parts / 152.0;
        double n = b <= per_sm ? (double)(long long)(b + 0.999) : b + 0.4;
        if (mixed && n > 1.0 && b <= per_sm) n -= 0.4;
        const double t = (n + lat) * (lz + 2 * r * halo);
        if (!best || t <= cost) {
            cost = t;
            best = lz;
        }
        if (parts == 1) break;
        lz = (nz + parts - 2) / (parts - 1);
    }
    if (cost_out) *cost_out = cost;
    return best;
}

// Which way a shell march goes.  Its tiles have rows along `row` (1: y, 2: z) and it advances along the other axis; a
// plane of the tile is a box of one node along that axis, so one tensor serves both (the shell is symmetric).
struct MarchAxes {
    int swap;        // 0: rows along y, march along z; 1: rows along z, march along y
    int rows, planes;  // the lattice's extents along them
    unsigned srow, splane;  // a node's distance to the next row and plane, in nodes
    long long prow, pplane;  // the same in the padded field
};
inline MarchAxes march_axes(const Grid &g, bool swap) {
    const long long pxy = (long long)g.px * g.py;
    const unsigned xy = (unsigned)g.nx * (unsigned)g.ny;
    return swap ? MarchAxes{1, g.nz, g.ny, xy, (unsigned)g.nx, pxy, g.px}
                : MarchAxes{0, g.ny, g.nz, (unsigned)g.nx, xy, g.px, pxy};
}

__device__ __forceinline__ long long march_pidx(const Grid &g, const MarchAxes &dir, int x, int y, int z) {
    return x + g.H + dir.prow * (y + g.H) + dir.pplane * (z + g.H);
}
// Offset of the force's component that the tile knows as c (0: x, 1: along its rows, 2: along the march).
__device__ __forceinline__ long long march_component(const Grid &g, const MarchAxes &dir, int c) {
    return g.N * (c == 0 ? 0 : (c == 1 ? 1 + dir.swap : 2 - dir.swap));
}

// Tensor maps of the shell fields of every ordered pair [a][b]: n_b and g_ab n_b (FP32: their deviations), boxes
// of the pair's diameter.
struct ShellMarchMaps {
    CUtensorMap n[MAXS * MAXS], gn[MAXS * MAXS];
};

// A mixture's blocks differ in length.  A.order lists the species with the smaller shells first; with few blocks
// the largest go first, so that the last to start are the short ones (128x32x32 channel, diameters 4 and 6: 46
// against 53 us; 90x75x66, diameters 2, 4, 6: 166 against 188 us).  Where many waves follow each other the order
// stays (512x128x128 channel: 1007 against 1029 us).
template <typename Args>
inline void march_order(Args &A, long long blocks, int per_sm) {
    if (blocks > 152ll * 2 * per_sm) return;
    for (int k = 0; 2 * k < A.M - 1; ++k) {
        const int t = A.order[k];
        A.order[k] = A.order[A.M - 1 - k];
        A.order[A.M - 1 - k] = t;
    }
}

}  // namespace lbe
