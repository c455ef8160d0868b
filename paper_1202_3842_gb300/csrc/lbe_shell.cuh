// Compile-time contact shells and the tile geometry of the shell-force kernel.
#pragma once

#include <utility>

namespace lbe {

// Contact shell of integer diameter S (Appendix, hard-sphere C^{alpha,mf}: the
// integral over unit vectors k^ at distance sigma becomes a sum over the lattice
// vectors e with S - 1/2 <= |e| < S + 1/2, i.e. S^2 - S + 1 <= |e|^2 <= S^2 + S).
__host__ __device__ constexpr bool in_shell(int S, int x, int y, int z) {
    int r2 = x * x + y * y + z * z;
    return r2 >= S * S - S + 1 && r2 <= S * S + S;
}
// sqrt of a positive integer at compile time: Newton's method started above
// the root, stopped when an iterate no longer decreases; the result is within
// one unit in the last place of the true root.
__host__ __device__ constexpr double ct_sqrt(double v) {
    double x = v > 1.0 ? v : 1.0;
    for (int i = 0; i < 200; ++i) {
        double nx = 0.5 * (x + v / x);
        if (!(nx < x)) break;
        x = nx;
    }
    return x;
}

// Column organisation of the half shell for the z-blocked kernels of the shell transpose: column
// pairs (ex, ey) / (-ex, -ey) with ex > 0 or (ex == 0, ey > 0); mask bit
// (ez + S) is set when (ex, ey, ez) lies in the shell.  The centre column
// (0, 0) holds ez = +-S only and is handled on its own.
__host__ __device__ constexpr int column_count(int S) {
    int c = 0;
    for (int y = -S; y <= S; ++y)
        for (int x = 0; x <= S; ++x) {
            if (!(x > 0 || y > 0)) continue;
            bool any = false;
            for (int z = -S; z <= S; ++z) any = any || in_shell(S, x, y, z);
            if (any) ++c;
        }
    return c;
}

template <int K>
struct Columns {
    int ex[K], ey[K];
    unsigned mask[K];
};

template <int S>
__host__ __device__ constexpr Columns<column_count(S)> make_columns() {
    Columns<column_count(S)> t{};
    int c = 0;
    for (int y = -S; y <= S; ++y)
        for (int x = 0; x <= S; ++x) {
            if (!(x > 0 || y > 0)) continue;
            unsigned m = 0;
            for (int z = -S; z <= S; ++z)
                if (in_shell(S, x, y, z)) m |= 1u << (z + S);
            if (m) {
                t.ex[c] = x;
                t.ey[c] = y;
                t.mask[c] = m;
                ++c;
            }
        }
    return t;
}

// Tile of the z-blocked shell transpose: 32 x TYB threads, TZ outputs per thread
// along z; the ring holds the 2S + TZ planes in use plus TZ in flight.
template <typename T, int S, int TZ, int TYB = 16>
struct ShellTileZ {
    static constexpr int A = 16 / (int)sizeof(T);
    static constexpr int TX = 32;
    static constexpr int TY = TYB;
    static constexpr int BX = ((TX + 2 * S + A - 1) + A - 1) / A * A;
    static constexpr int BY = TY + 2 * S;
    static constexpr int R = 2 * S + 2 * TZ;
    static constexpr int PLANE = BX * BY;
    static constexpr int PLANE_BYTES = ((PLANE * (int)sizeof(T)) + 127) / 128 * 128;
    static constexpr int SLOT_BYTES = 2 * PLANE_BYTES;
    static constexpr int SMEM = R * SLOT_BYTES + 256 + 128;
    static constexpr int LZ = TZ == 3 ? 18 : 16;  // planes per CTA, a multiple of TZ
};

// Tile of the FP32 z-blocked shell transpose on the interleaved field: one
// 8-byte element (Lambda, g Lambda) per node, so one shared load fetches both
// values of a stencil point and the two sums run as packed f32x2 arithmetic.
// TMA sees 8-byte elements: the x coordinate must be even (A = 2).
template <int S, int TZ, int TYB = 16>
struct ShellTileZ2 {
    static constexpr int A = 2;
    static constexpr int TX = 32;
    static constexpr int TY = TYB;
    static constexpr int BX = ((TX + 2 * S + A - 1) + A - 1) / A * A;
    static constexpr int BY = TY + 2 * S;
    static constexpr int R = 2 * S + 2 * TZ;
    static constexpr int PLANE = BX * BY;  // 8-byte elements of one plane
    static constexpr int PLANE_BYTES = ((PLANE * 8) + 127) / 128 * 128;
    static constexpr int SLOT_BYTES = PLANE_BYTES;
    static constexpr int SMEM = R * SLOT_BYTES + 256 + 128;
    static constexpr int LZ = (16 + TZ - 1) / TZ * TZ;  // planes per CTA, a multiple of TZ
};

}  // namespace lbe
