// Sums of FP64 populations on the integer pipe.  GB300 adds two doubles per clock and SM, but 64-bit integers at a
// quarter of the FP32 rate or more, so the moments of a node (57 of K4's 300 FP64 instructions per node and species, all
// of K1's) are summed in block floating point: the values as 64-bit integers in units of 2^-58 of the power of two
// above the largest, added exactly, and the sum rounded once to a double.  A value is rounded to the unit, a 32nd of
// the largest value's last bit, so the sum's error is below that of the FP64 additions it replaces (1.1e-16 of the
// sum against 5.4e-16, worst of 4000 draws).  Infinities, NaN and exponents at either end of the range take those additions.
// K4 of the 256x64x64 channel 1197 -> 987 us, K1 92 -> 88; K4 of the 48^3 well with SD-TR 53 -> 46 us.
#pragma once
#include <cstring>

#include "lbe_device.cuh"

namespace lbe {

__host__ __device__ __forceinline__ long long double_bits(double v) {
#ifdef __CUDA_ARCH__
    return __double_as_longlong(v);
#else
    long long b;
    std::memcpy(&b, &v, 8);
    return b;
#endif
}
__host__ __device__ __forceinline__ double bits_double(long long b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double(b);
#else
    double v;
    std::memcpy(&v, &b, 8);
    return v;
#endif
}

// 2 v by its exponent; zero, subnormal and the largest values, whose exponents do not tell, by shifting their bits.
// (An addition there was executed for every value: K4 of the 256x64x64 channel 861 -> 919 us.)
__host__ __device__ __forceinline__ double twice(double v) {
    const long long b = double_bits(v), sign = (long long)0x8000000000000000ull;
    const unsigned e = (unsigned)(b >> 52) & 0x7ffu;
    if (e - 1u < 0x7fdu) return bits_double(b + (1ll << 52));
    if (e == 0u) return bits_double((b & sign) | ((b << 1) & ~sign));
    return e == 0x7feu ? bits_double((b & sign) | 0x7ff0000000000000ll) : v;
}

// Largest biased exponent of the populations, or 0 where they cannot be summed as integers.
__host__ __device__ __forceinline__ int block_exponent(const double *v) {
    unsigned m = 0;
#pragma unroll
    for (int p = 0; p < Q; ++p) {
        const unsigned h = (unsigned)(double_bits(v[p]) >> 32) & 0x7fffffffu;
        m = h > m ? h : m;
    }
    const int e = (int)(m >> 20);
    return e >= 64 && e < 2040 ? e : 0;
}
// v 2^(1080 - emax), rounded: at most 2^58
__host__ __device__ __forceinline__ long long to_block(double v, int emax) {
    const long long b = double_bits(v);
    const int sh = emax - ((int)(b >> 52) & 0x7ff);  // (a subnormal value is far below the unit)
    const unsigned long long m = ((unsigned long long)b & 0xfffffffffffffull) | 0x10000000000000ull;
    const long long r = (long long)(((m << 6 >> (sh < 63 ? sh : 63)) + 1) >> 1);
    return b < 0 ? -r : r;
}
// s 2^(emax - 1080), to nearest even; |s| < 2^63
__host__ __device__ __forceinline__ double from_block(long long s, int emax) {
    if (s == 0) return 0.0;
    unsigned long long a = (unsigned long long)(s < 0 ? -s : s);
#ifdef __CUDA_ARCH__
    const int lz = __clzll((long long)a);
#else
    const int lz = __builtin_clzll(a);
#endif
    a <<= lz;
    // the mantissa's leading bit adds one to the exponent field, and so does a carry out of it
    unsigned long long r = ((unsigned long long)(emax + 5 - lz) << 52) + (a >> 11);
    r += ((a & 0x7ff) + ((a >> 11) & 1)) > 0x400 ? 1 : 0;
    return bits_double((long long)(r | ((unsigned long long)s & 0x8000000000000000ull)));
}

// Sum of the populations.
__host__ __device__ __forceinline__ double block_sum(const double *f) {
    const int e = block_exponent(f);
    if (e == 0) {
        double n = f[0];
#pragma unroll
        for (int p = 1; p < Q; ++p) n += f[p];
        return n;
    }
    long long n = to_block(f[0], e);
#pragma unroll
    for (int p = 1; p < Q; ++p) n += to_block(f[p], e);
    return from_block(n, e);
}
// Sum and first moment.
__host__ __device__ __forceinline__ void block_moments(const double *g, double &Pi, double J[3]) {
    const int e = block_exponent(g);
    if (e == 0) {
        double s = g[0], d[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            s += g[1 + 2 * k] + g[2 + 2 * k];
            d[k] = g[1 + 2 * k] - g[2 + 2 * k];
        }
        Pi = s;
        J[0] = d[0] + d[3] + d[4] + d[5] + d[6];
        J[1] = d[1] + d[3] - d[4] + d[7] + d[8];
        J[2] = d[2] + d[5] - d[6] + d[7] - d[8];
        return;
    }
    long long s = to_block(g[0], e), j[3] = {0, 0, 0};
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        // pairs: x, y, z; (1,1,0), (1,-1,0), (1,0,1), (1,0,-1), (0,1,1), (0,1,-1)
        const long long a = to_block(g[1 + 2 * k], e), b = to_block(g[2 + 2 * k], e), d = a - b;
        s += a + b;
        if (k == 0 || (k >= 3 && k < 7)) j[0] += d;
        if (k == 1 || k == 3 || k == 7 || k == 8) j[1] += d;
        if (k == 4) j[1] -= d;
        if (k == 2 || k == 5 || k == 7) j[2] += d;
        if (k == 6 || k == 8) j[2] -= d;
    }
    Pi = from_block(s, e);
#pragma unroll
    for (int c = 0; c < 3; ++c) J[c] = from_block(j[c], e);
}

}  // namespace lbe
