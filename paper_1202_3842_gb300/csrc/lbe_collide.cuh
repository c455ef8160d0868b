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
// below).  That is 14 flops per population where each population's own f_eq, S_f and update took 36.
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
    T kf, kg, k2, omc;
    T ua[3], u[3], X9[3], G9[3], Of[3], Og[3];

    // dn, Pi: n and Pi, or their deviations from n0 when the populations are deviations from w_p n0; in0 = 1/n0
    // (UNIT only)
    __device__ __forceinline__ void set(T n, T dn, T Pi, const T *ua_, const T *u_, const T *C, const T *nF, T om,
                                        T inv, T in0) {
        const T w = UNIT ? in0 : (T)(1.0 / 36.0), wom = w * om, winv = w * inv;
        const T uau = ua_[0] * u_[0] + ua_[1] * u_[1] + ua_[2] * u_[2];
        const T uu = u_[0] * u_[0] + u_[1] * u_[1] + u_[2] * u_[2];
        const T iso = (T)1.5 * n * ((T)2 * uau - uu);
        T s0 = (T)0;
        const T a = (T)3 * wom * n, b = (T)3 * winv;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const T X = C[c] + nF[c], m = a * ua_[c], bX = b * X, bY = b * nF[c];
            ua[c] = ua_[c];
            u[c] = u_[c];
            s0 = c == 0 ? bX * ua_[0] : s0 + bX * ua_[c];
            X9[c] = (T)3 * bX;
            G9[c] = (T)3 * (bX + b * C[c]);  // inv (18 C + 9 nF) / 36
            Of[c] = m + bX;
            Og[c] = m + bY;
        }
        kf = wom * (dn - iso) - s0;
        kg = wom * (Pi - iso) - s0;
        k2 = (T)4.5 * wom * n;
        omc = (T)1 - om;
    }

    // the rest populations (G false: f only)
    template <bool G = true>
    __device__ __forceinline__ void rest(T &f, T &g) const {
        f = UNIT ? omc * f + kf : omc * f + (T)12 * kf;
        if constexpr (G) g = UNIT ? omc * g + kg : omc * g + (T)12 * kg;
    }
    // the populations of the pair P, P + 1 = opposite of P
    template <int P, bool G = true>
    __device__ __forceinline__ void pair(T &fp, T &fm, T &gp, T &gm) const {
        static_assert(P % 2 == 1 && P < Q, "first population of a pair");
        const T s = link_dot<T, P>(ua), t = link_dot<T, P>(u);
        const T h = ((T)2 * s - t) * t;
        const T ef = link_dot<T, P>(X9) * s + (k2 * h + kf), of = link_dot<T, P>(Of);
        constexpr T wp = (T)(!UNIT && P < 7 ? 2 : 1);  // axis links: weight 1/18
        fp = omc * fp + wp * (ef + of);
        fm = omc * fm + wp * (ef - of);
        if constexpr (G) {
            const T eg = link_dot<T, P>(G9) * s + (k2 * h + kg), og = link_dot<T, P>(Og);
            gp = omc * gp + wp * (eg + og);
            gm = omc * gm + wp * (eg - og);
        }
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
