// The collision of one species at one node (Sec. "Hard sphere fluid mixture in a potential well"), shared by K4
// and the scheme ablations.  With v_T^2 = 1/3 the Hermite contractions expand to
//   f_eq = w [A + 3 n c.u^a + (9/2) n (2 c.u^a - c.u) c.u],        A = n - iso   (g_eq: B = Pi - iso),
//   iso  = (3/2) n (2 u^a.u - u.u),
//   S_f  = w [s0 + 3 c.X + 9 (c.X)(c.u^a)],                        X = C + nF, s0 = -3 X.u^a,
//   S_g  = w [s0 + 3 c.Y + (18 c.C + 9 c.Y)(c.u^a)],               Y = nF,
//   f*   = (1 - om) f + om f_eq + inv S_f                          (g the same).
// Everything but (1 - om) f is, for the two populations of an opposite pair, a part even in c plus or minus a part
// odd in c:
//   even_f = kf + k2 (2s - t) t + (c.X9) s,  even_g = kg + k2 (2s - t) t + (c.G9) s,  s = c.u^a, t = c.u,
//   odd_f  = c.Of,  odd_g = c.Og,
// so a pair shares its dot products, and the constants carry om, inv and the edge links' weight 1/36 (or 1/n0,
// below).  That is 24 operations for the four populations of an edge pair, f and g, where one population's own f_eq,
// S_f and update took 36 flops.
#pragma once
#include <type_traits>
#include <utility>

#include "lbe_block_sum.cuh"
#include "lbe_device.cuh"

namespace lbe {

// c_p . v; a sum never starts from 0 (0 + v is an addition in IEEE arithmetic).
template <typename T, int P>
__device__ __forceinline__ T link_dot(const T *v) {
    constexpr int c[3] = {cx(P), cy(P), cz(P)};
    constexpr int i = c[0] != 0 ? 0 : (c[1] != 0 ? 1 : 2);
    constexpr int j = c[2] != 0 && i != 2 ? 2 : (c[1] != 0 && i != 1 ? 1 : -1);
    const T a = c[i] > 0 ? v[i] : -v[i];
    if constexpr (j < 0)
        return a;
    else
        return c[j] > 0 ? a + v[j] : a - v[j];
}

// Populations in the units they are stored in (Store::load_unit): with 16 bits, UNIT, s = d / (w_p n0), so that a sum
// over populations weighs them by w_p (in units of the edge links' 1/36) and the collision's even and odd parts lose
// the weight; no population is then multiplied by w_p n0 on its way in or out.

// Sum of the populations (UNIT: of 36 w_p s_p).
template <bool UNIT, typename T>
__device__ __forceinline__ T zeroth_moment(const T *f) {
    if constexpr (UNIT) {
        T a = f[1], e = f[7];
#pragma unroll
        for (int p = 2; p < 7; ++p) a += f[p];
#pragma unroll
        for (int p = 8; p < Q; ++p) e += f[p];
        return (T)12 * f[0] + ((T)2 * a + e);
    } else if constexpr (std::is_same_v<T, double>) {
        return block_sum(f);
    } else {
        T n = f[0];
#pragma unroll
        for (int p = 1; p < Q; ++p) n += f[p];
        return n;
    }
}
// Sum and first moment (UNIT: of 36 w_p s_p) from the sums and differences of opposite pairs.
template <bool UNIT, typename T>
__device__ __forceinline__ void pair_moments(const T *g, T &Pi, T J[3]) {
    if constexpr (std::is_same_v<T, double>) {
        block_moments(g, Pi, J);
        return;
    }
    // pairs: x, y, z; (1,1,0), (1,-1,0), (1,0,1), (1,0,-1), (0,1,1), (0,1,-1)
    T d[9], s = UNIT ? g[1] + g[2] : g[0];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        if constexpr (UNIT) {
            if (k == 3) s = (T)2 * s + (T)12 * g[0];
            if (k > 0) s += g[1 + 2 * k] + g[2 + 2 * k];
        } else {
            s += g[1 + 2 * k] + g[2 + 2 * k];
        }
        d[k] = g[1 + 2 * k] - g[2 + 2 * k];
        if (UNIT && k < 3) d[k] *= (T)2;
    }
    Pi = s;
    J[0] = d[0] + d[3] + d[4] + d[5] + d[6];
    J[1] = d[1] + d[3] - d[4] + d[7] + d[8];
    J[2] = d[2] + d[5] - d[6] + d[7] - d[8];
}

// The density of pulled populations (shifted storage: n0 plus the sum of the deviations).
template <typename S, typename T>
__device__ __forceinline__ T density_of(const T *v, T n0) {
    constexpr bool UNIT = sizeof(S) == 2;
    const T n = zeroth_moment<UNIT>(v);
    if constexpr (UNIT) return n0 + (T)(1.0 / 36.0) * n0 * n;
    return Store<S, T>::shifted ? n0 + n : n;
}

template <typename T, bool UNIT = false>
struct Collision {
    T kf, kg, k2, rel;
    T ua[3], u[3], X9[3], G9[3], Of[3], Og[3];

    // dn, Pi: n and Pi, or their deviations from n0 when the populations are deviations from w_p n0; in0 = 1/n0
    // (UNIT only)
    __device__ __forceinline__ void set(T n, T dn, T Pi, const T *J, const T *ua_, const T *u_, const T *C,
                                        const T *nF, T om, T inv, T in0) {
        // Every step scales a node's density by 36 times the factor `share` and its momentum by 12 times `share3`, so what
        // a rounded constant om / 36 is off (up to 5e-8), or 1 - om for om < 1/2, would add up from step to step: the
        // factors are in two parts, the momentum enters as J and not as n u^a, and relax() takes om.  What is left
        // is the values' own rounding.  Momentum of a 16^3 gas in uniform flow after 1000 steps, relative change: 6e-5
        // with rounded constants, 1.6e-6 now (tau 0.7; 1.3e-5 where each population had its own f_eq); velocity of
        // the 512x128x128 channel after 40 steps, error against 64 bits: 7.4e-7, 1.8e-7 now (5.2e-7).  K4 keeps its
        // time (hbm bound).
        constexpr T w36 = (T)(1.0 / 36.0), w36_lo = (T)(1.0 / 36.0 - (double)w36);
        constexpr T w12 = (T)(1.0 / 12.0), w12_lo = (T)(1.0 / 12.0 - (double)w12);
        const T wom = in0 * om, winv = (UNIT ? in0 : w36) * inv;
        const auto share = [&](T v) { return UNIT ? wom * v : om * (w36 * v + w36_lo * v); };  // v om / 36
        const auto share3 = [&](T v) { return UNIT ? (T)3 * wom * v : om * (w12 * v + w12_lo * v); };
        const T uau = ua_[0] * u_[0] + ua_[1] * u_[1] + ua_[2] * u_[2];
        const T uu = u_[0] * u_[0] + u_[1] * u_[1] + u_[2] * u_[2];
        const T iso = (T)1.5 * n * ((T)2 * uau - uu);
        T s0 = (T)0;
        const T a = share3(n), b = (T)3 * winv;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            // (no density: no equilibrium, whatever g's momentum)
            const T X = C[c] + nF[c], m = share3(n > (T)0 ? J[c] : (T)0), bX = b * X, bY = b * nF[c];
            ua[c] = ua_[c];
            u[c] = u_[c];
            s0 = c == 0 ? bX * ua_[0] : s0 + bX * ua_[c];
            X9[c] = (T)3 * bX;
            G9[c] = (T)3 * (bX + b * C[c]);  // inv (18 C + 9 nF) / 36
            Of[c] = m + bX;
            Og[c] = m + bY;
        }
        kf = share(dn - iso) - s0;
        kg = share(Pi - iso) - s0;
        k2 = (T)1.5 * a;
        rel = UNIT ? (T)1 - om : om;
    }
    // (1 - om) f + part
    __device__ __forceinline__ T relax(T f, T part) const {
        return UNIT ? rel * f + part : f + (part - rel * f);
    }

    // the rest populations
    __device__ __forceinline__ void rest(T &f, T &g) const {
        f = relax(f, UNIT ? kf : (T)12 * kf);
        g = relax(g, UNIT ? kg : (T)12 * kg);
    }
    // the populations of the pair P, P + 1 = opposite of P
    template <int P>
    __device__ __forceinline__ void pair(T &fp, T &fm, T &gp, T &gm) const {
        static_assert(P % 2 == 1 && P < Q, "first population of a pair");
        const T s = link_dot<T, P>(ua), t = link_dot<T, P>(u);
        const T h = ((T)2 * s - t) * t;
        const T ef = link_dot<T, P>(X9) * s + (k2 * h + kf), of = link_dot<T, P>(Of);
        const T eg = link_dot<T, P>(G9) * s + (k2 * h + kg), og = link_dot<T, P>(Og);
        constexpr T wp = (T)(!UNIT && P < 7 ? 2 : 1);  // axis links: weight 1/18
        fp = relax(fp, wp * (ef + of));
        fm = relax(fm, wp * (ef - of));
        gp = relax(gp, wp * (eg + og));
        gm = relax(gm, wp * (eg - og));
    }
};

// The same for FP64 populations, where every operation counts (GB300 has two FP64 lanes per SM): the even part of a pair is a
// quadratic form in c,
//   k + c.Q.c,  Q_ij = k2 (2u^a - u)_i u_j + X9_i u^a_j  (symmetric part),
// so an axis takes k + Q_ii, an edge k + Q_ii + Q_jj +- 2 Q_ij, and with iso and s0 the constants are
//   kf = w om n - tr(Q) / 3,  kg = w om Pi - tr(Q) / 3.
// One distribution at a time, g's form from f's (G9 - X9 = 3 b C): about 200 FP64 instructions per node and species
// besides the moments instead of 243.  K4 of the 256x64x64 channel 989 -> 811 us, of the 48^3 well with SD-TR 47 -> 38.
struct Collision64 {
    double k, omc, q[3], r[3], o[3];  // r: 2 Q_xy, 2 Q_xz, 2 Q_yz; o: odd part
    double kg, og[3], d[3], ua[3];    // what next() needs

    __device__ __forceinline__ void set(double n, double Pi, const double *ua_, const double *u, const double *C,
                                        const double *nF, double om, double inv) {
        const double wom = 1.0 / 36.0 * om, a = 3.0 * wom * n, b = 3.0 / 36.0 * inv, k2 = 4.5 * wom * n;
        double v[3], X9[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double m = a * ua_[c], bX = b * (C[c] + nF[c]);
            ua[c] = ua_[c];
            v[c] = k2 * (2.0 * ua[c] - u[c]);
            X9[c] = 3.0 * bX;
            d[c] = 3.0 * b * C[c];
            o[c] = m + bX;
            og[c] = m + b * nF[c];
            q[c] = v[c] * u[c] + X9[c] * ua[c];
        }
#pragma unroll
        for (int e = 0; e < 3; ++e) {
            const int i = e == 2 ? 1 : 0, j = e == 0 ? 1 : 2;
            r[e] = v[i] * u[j] + v[j] * u[i] + X9[i] * ua[j] + X9[j] * ua[i];
        }
        const double tr = q[0] + q[1] + q[2];
        k = wom * n - 1.0 / 3.0 * tr;
        kg = wom * Pi - 1.0 / 3.0 * tr;
        omc = 1.0 - om;
    }
    // from f to g
    __device__ __forceinline__ void next() {
        k = kg;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            o[c] = og[c];
            q[c] += d[c] * ua[c];
        }
#pragma unroll
        for (int e = 0; e < 3; ++e) {
            const int i = e == 2 ? 1 : 0, j = e == 0 ? 1 : 2;
            r[e] += d[i] * ua[j] + d[j] * ua[i];
        }
    }
    __device__ __forceinline__ void rest(double &f) const { f = omc * f + 12.0 * k; }
    template <int P>
    __device__ __forceinline__ void pair(double &fp, double &fm) const {
        if constexpr (P < 7) {  // axis links: weight 1/18
            constexpr int i = (P - 1) / 2;
            const double e = k + q[i];
            fp = omc * fp + twice(e + o[i]);
            fm = omc * fm + twice(e - o[i]);
        } else {
            constexpr int i = cx(P) ? 0 : 1, j = cz(P) ? 2 : 1;
            constexpr bool same = (i == 0 ? cx(P) : cy(P)) * (j == 1 ? cy(P) : cz(P)) > 0;
            static_assert((i == 0 ? cx(P) : cy(P)) == 1, "first population of a pair");
            const double t = (k + q[i]) + q[j], e = same ? t + r[i + j - 1] : t - r[i + j - 1];
            const double h = same ? o[i] + o[j] : o[i] - o[j];
            fp = omc * fp + (e + h);
            fm = omc * fm + (e - h);
        }
    }
    __device__ __forceinline__ void all(double *v) const {
        rest(v[0]);
        [&]<int... K>(std::integer_sequence<int, K...>) {
            (pair<2 * K + 1>(v[2 * K + 1], v[2 * K + 2]), ...);
        }(std::make_integer_sequence<int, 9>{});
    }
};

// The same collision with every population's f_eq, S_f and update on its own, on the populations themselves (the
// order in which FP32 runs of three and four species round; see k_collide_pair).
template <typename T>
__device__ __forceinline__ void ordered_momentum(const T *g, T J[3]) {
    J[0] = J[1] = J[2] = (T)0;
#pragma unroll
    for (int p = 1; p < Q; ++p) {
        if (cx(p)) J[0] += (T)cx(p) * g[p];
        if (cy(p)) J[1] += (T)cy(p) * g[p];
        if (cz(p)) J[2] += (T)cz(p) * g[p];
    }
}
template <typename T>
__device__ __forceinline__ void collide_whole(T n, T Pi, const T *ua, const T *u, const T *C, const T *nF, T om,
                                              T inv, T *f, T *g) {
    const T uau = ua[0] * u[0] + ua[1] * u[1] + ua[2] * u[2];
    const T uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    const T iso = (T)1.5 * n * ((T)2 * uau - uu);
    const T A = n - iso, B = Pi - iso;
    T X[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) X[c] = C[c] + nF[c];
    const T sf0 = (T)-3 * (X[0] * ua[0] + X[1] * ua[1] + X[2] * ua[2]);
    [&]<int... P>(std::integer_sequence<int, P...>) {
        (
            [&] {
                constexpr T w = (T)wq(P);
                T cua = 0, cu = 0, cX = 0, cY = 0, cC = 0;
                if constexpr (P > 0) {
                    cua = link_dot<T, P>(ua);
                    cu = link_dot<T, P>(u);
                    cX = link_dot<T, P>(X);
                    cY = link_dot<T, P>(nF);
                    cC = link_dot<T, P>(C);
                }
                const T t1 = (T)3 * n * cua + (T)4.5 * n * ((T)2 * cua * cu - cu * cu);
                const T feq = w * (A + t1);
                const T geq = w * (B + t1);
                const T Sf = w * (sf0 + (T)3 * cX + (T)9 * cX * cua);
                const T Sg = w * (sf0 + (T)3 * cY + (T)18 * cC * cua + (T)9 * cY * cua);
                f[P] = f[P] + om * (feq - f[P]) + inv * Sf;
                g[P] = g[P] + om * (geq - g[P]) + inv * Sg;
            }(),
            ...);
    }(std::make_integer_sequence<int, Q>{});
}

}  // namespace lbe
