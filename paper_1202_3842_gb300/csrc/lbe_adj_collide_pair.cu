// K4 transposed for one or two species (the arithmetic of k_adj_collide + k_adj_write in lbe_adjoint.cu, opposite
// populations together).
//
// Two species: the layout of the forward collision (lbe_collide_pair.cu), warps 0 - 3 of a 256-thread CTA with species
// 0 and warps 4 - 7 with species 1 of the same 128 nodes (one species: one thread per node).  Each thread
//   pass A  pulls its own species' populations and forms its moments; n and J of the partner species, through
//           shared memory, give the barycentric u;
//   pass B  push-gathers the adjoint of its post-collision populations (kept in registers) and transposes the
//           collision; the adjoint of u is the sum over both species, again by one exchange with the partner;
//   pass C  transposes the moment recovery, adds lambda_F, writes lambda_C and the adjoint of its pre-collision
//           populations.
// Cross-species sums are formed in species order (0 then 1), as in the one-thread-per-node kernel.
// A warp none of whose nodes has a blocked link pulls and gathers without the bounce-back selects, as the forward
// kernels do.  In pass B the two populations of an opposite pair share their dot products and enter as the sum E and
// the difference D of their adjoints.
// Bounds: latency of the pulls and gathers (38 loads each pass); three CTAs per SM in FP32 hide more of it than two
// (gradient of 20 steps of the 256x64x64 channel, FP32: 30.7 ms with a second pull of the populations instead of
// registers, 30.5 with registers and two CTAs, 29.0 with three).
#include <type_traits>
#include <utility>

#include "lbe_collide.cuh"
#include "lbe_device.cuh"
#include "lbe_launch.h"
#include "lbe_node.cuh"

namespace lbe {

constexpr int ACP = 256;  // threads per CTA: 128 nodes (two species) or 256 (one)

// adjoint of the post-collision population p (streaming transposed), density adjoint added for f
template <typename T, int P, bool SEL>
__device__ __forceinline__ T gather_post_pair(const T *__restrict__ lY, const T *__restrict__ ln, long long N,
                                              long long i, const NbrOff &o, uint32_t m) {
    if constexpr (SEL) {
        if (m & (1u << opp(P))) {
            const T v = lY[(long long)opp(P) * N + i];
            return ln ? v + ln[i] : v;
        }
    }
    const long long j = i + src_off<opp(P)>(o);  // r + c_P
    const T v = lY[(long long)P * N + j];
    return ln ? v + ln[j] : v;
}

// Values of the partner species at the same node, through shared memory; the two warps over the same 32 nodes wait
// for each other at named barrier 1 + w.  Every thread takes part.
template <typename T, int M, int K>
__device__ __forceinline__ void partners(T (*xch)[K][128], int a, int loc, const T (&v)[K], T (&p)[K]) {
    if constexpr (M == 2) {
#pragma unroll
        for (int k = 0; k < K; ++k) xch[a][k][loc] = v[k];
        asm volatile("bar.sync %0, 64;" ::"r"(1 + (loc >> 5)) : "memory");
#pragma unroll
        for (int k = 0; k < K; ++k) p[k] = xch[1 - a][k][loc];
    } else {
#pragma unroll
        for (int k = 0; k < K; ++k) p[k] = (T)0;
    }
}

template <typename S, typename T, int M>
__global__ void __launch_bounds__(ACP, sizeof(T) == 4 ? 3 : 1)
    k_adj_collide_pair(Grid g, const S *__restrict__ post, const uint32_t *__restrict__ mask,
                       const T *__restrict__ C, const T *__restrict__ F, AdjParams ap, const T *__restrict__ lYf_in,
                       const T *__restrict__ lYg_in, const T *__restrict__ lnd_in, T *__restrict__ lYf_out,
                       T *__restrict__ lYg_out, T *__restrict__ lC, T *__restrict__ lF) {
    static_assert(M == 1 || M == 2, "one or two species");
    __shared__ T xa[M][4][128], xb[M][3][128];
    const int a = M == 2 ? (int)(threadIdx.x >> 7) : 0;
    const int loc = M == 2 ? (int)(threadIdx.x & 127) : 0;
    const long long i = M == 2 ? (long long)blockIdx.x * (ACP / 2) + loc : (long long)blockIdx.x * ACP + threadIdx.x;
    const bool valid = i < g.N;
    int x = 0, y = 0, z = 0;
    if (valid) node_xyz(g, i, x, y, z);
    const uint32_t m = valid ? mask[i] : 1u;
    const bool fluid = !(m & 1u);
    const bool plain = __all_sync(0xffffffffu, (m >> 1) == 0u);
    const double n0d = a == 0 ? ap.sp[0].n0 : ap.sp[1].n0;
    const T om = (T)(a == 0 ? ap.sp[0].omega_eff : ap.sp[1].omega_eff);
    const T inv = (T)(a == 0 ? ap.sp[0].inv : ap.sp[1].inv);
    NbrOff o{};
    if (fluid) o = nbr_offsets(g, x, y, z);

    // ---- pass A: forward moments of this species
    T n = 0, inv_n = 0, J[3] = {0, 0, 0}, ua[3] = {0, 0, 0}, Cv[3] = {0, 0, 0}, Fv[3] = {0, 0, 0};
    T nF[3] = {0, 0, 0};
    T lf[Q], lg[Q];
    if (fluid) {
        const T n0 = (T)n0d;
        const S *fb = post + pop_off(a, 0, 0, g.N);
        const S *gb = post + pop_off(a, 1, 0, g.N);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            Cv[c] = C[((long long)a * 3 + c) * g.N + i];
            Fv[c] = F[((long long)a * 3 + c) * g.N + i];
        }
        T Jt[3] = {0, 0, 0};
        auto moments = [&](auto Sel) {
            constexpr bool SEL = decltype(Sel)::value;
            T f[Q], gq[Q];
            [&]<int... P>(std::integer_sequence<int, P...>) {
                ((f[P] = pull<S, T, P, SEL>(fb, g.N, i, o, m, n0)), ...);
                ((gq[P] = pull<S, T, P, SEL>(gb, g.N, i, o, m, n0)), ...);
            }(std::make_integer_sequence<int, Q>{});
            n = zeroth_moment<false>(f);
            ordered_momentum(gq, Jt);
        };
        if (plain)
            moments(std::false_type{});
        else
            moments(std::true_type{});
        inv_n = n > (T)0 ? (T)1 / n : (T)0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            nF[c] = n * Fv[c];
            J[c] = ap.consistent ? Jt[c] + (T)0.5 * nF[c] : Jt[c] + (T)0.5 * (Cv[c] + nF[c]);
            ua[c] = J[c] * inv_n;
        }
        // the gather's loads are issued before the exchange
        const T *lYf = lYf_in + (long long)a * Q * g.N;
        const T *lYg = lYg_in + (long long)a * Q * g.N;
        const T *lnd = lnd_in + (long long)a * g.N;
        auto gather = [&](auto Sel) {
            constexpr bool SEL = decltype(Sel)::value;
            [&]<int... P>(std::integer_sequence<int, P...>) {
                ((lf[P] = gather_post_pair<T, P, SEL>(lYf, lnd, g.N, i, o, m)), ...);
                ((lg[P] = gather_post_pair<T, P, SEL>(lYg, nullptr, g.N, i, o, m)), ...);
            }(std::make_integer_sequence<int, Q>{});
        };
        if (plain)
            gather(std::false_type{});
        else
            gather(std::true_type{});
    }
    const T va[4] = {n, J[0], J[1], J[2]};
    T pa[4];
    partners<T, M, 4>(xa, a, loc, va, pa);
    const T ntot = a == 0 ? n + pa[0] : pa[0] + n;
    const T inv_tot = ntot > (T)0 ? (T)1 / ntot : (T)0;
    T u[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) u[c] = (a == 0 ? J[c] + pa[c + 1] : pa[c + 1] + J[c]) * inv_tot;
    const T uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];

    // ---- pass B: collision transposed
    T lu[3] = {0, 0, 0}, lua[3] = {0, 0, 0}, lCs[3] = {0, 0, 0}, lnFs[3] = {0, 0, 0}, lns = 0, lPis = 0;
    if (fluid) {
        const T uau = ua[0] * u[0] + ua[1] * u[1] + ua[2] * u[2];
        T X[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) X[c] = Cv[c] + nF[c];
        constexpr T w0 = (T)wq(0);
        T lA = w0 * om * lf[0], lB = w0 * om * lg[0], lsf0 = w0 * inv * (lf[0] + lg[0]), lnv = 0;
        T lX[3] = {0, 0, 0}, lnFv[3] = {0, 0, 0}, lCv[3] = {0, 0, 0}, luav[3] = {0, 0, 0}, lua_u[3] = {0, 0, 0};
        [&]<int... KP>(std::integer_sequence<int, KP...>) {
            (
                [&] {
                    constexpr int P = 2 * KP + 1;  // and its opposite, P + 1
                    constexpr T w = (T)wq(P);
                    const T wom = w * om, winv = w * inv;
                    const T Ef = lf[P] + lf[P + 1], Df = lf[P] - lf[P + 1];
                    const T Eg = lg[P] + lg[P + 1], Dg = lg[P] - lg[P + 1];
                    const T H = wom * (Ef + Eg), K = wom * (Df + Dg);
                    const T s = link_dot<T, P>(ua), t = link_dot<T, P>(u);
                    const T cX = link_dot<T, P>(X), cY = link_dot<T, P>(nF), cC = link_dot<T, P>(Cv);
                    lA += wom * Ef;
                    lB += wom * Eg;
                    lsf0 += winv * (Ef + Eg);
                    const T lcX = winv * ((T)3 * Df + (T)9 * s * Ef);
                    const T lcY = winv * ((T)3 * Dg + (T)9 * s * Eg);
                    const T lcC = (T)18 * winv * s * Eg;
                    const T lcua = winv * ((T)9 * cX * Ef + ((T)18 * cC + (T)9 * cY) * Eg) +
                                   n * ((T)3 * K + (T)9 * t * H);
                    const T lcu = (T)9 * n * (s - t) * H;
                    lnv += (T)3 * s * K + (T)4.5 * ((T)2 * s - t) * t * H;
                    auto add = [&](auto Cc) {
                        constexpr int c = decltype(Cc)::value;
                        constexpr int cc = c == 0 ? cx(P) : (c == 1 ? cy(P) : cz(P));
                        if constexpr (cc != 0) {
                            luav[c] += (T)cc * lcua;
                            lua_u[c] += (T)cc * lcu;
                            lX[c] += (T)cc * lcX;
                            lnFv[c] += (T)cc * lcY;
                            lCv[c] += (T)cc * lcC;
                        }
                    };
                    add(std::integral_constant<int, 0>{});
                    add(std::integral_constant<int, 1>{});
                    add(std::integral_constant<int, 2>{});
                }(),
                ...);
        }(std::make_integer_sequence<int, 9>{});
        // sf0 = -3 X.u^a ; X = C + nF ; A = n - iso ; B = Pi - iso ; iso = 1.5 n (2 u^a.u - u.u)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            lX[c] += (T)-3 * ua[c] * lsf0;
            luav[c] += (T)-3 * X[c] * lsf0;
            lCv[c] += lX[c];
            lnFv[c] += lX[c];
        }
        const T liso = -lA - lB;
        lnv += lA + (T)1.5 * ((T)2 * uau - uu) * liso;
        const T luau = (T)3 * n * liso;
        const T luu = (T)-1.5 * n * liso;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            luav[c] += u[c] * luau;
            lu[c] += lua_u[c] + ua[c] * luau + (T)2 * u[c] * luu;
            lua[c] = luav[c];
            lCs[c] = lCv[c];
            lnFs[c] = lnFv[c];
        }
        lns = lnv;
        lPis = lB;
    }
    // ---- u = sum J / sum n: the adjoint of u summed over both species (species order)
    T lJtot[3] = {0, 0, 0}, lntot = 0, pb[3];
    partners<T, M, 3>(xb, a, loc, lu, pb);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const T lp = pb[c];
        const T lut = a == 0 ? lu[c] + lp : lp + lu[c];
        if (ntot > (T)0) {
            lJtot[c] = lut * inv_tot;
            lntot -= lut * u[c] * inv_tot;
        }
    }
    if (!valid) return;
    T *of = lYf_out + (long long)a * Q * g.N + i;
    T *og = lYg_out + (long long)a * Q * g.N + i;
    if (!fluid) {
#pragma unroll
        for (int c = 0; c < 3; ++c) lC[((long long)a * 3 + c) * g.N + i] = (T)0;
#pragma unroll
        for (int p = 0; p < Q; ++p) {
            of[(long long)p * g.N] = (T)0;
            og[(long long)p * g.N] = (T)0;
        }
        return;
    }
    // ---- pass C: moment recovery transposed, outputs
    const int coord = ap.axis == 0 ? x : (ap.axis == 1 ? y : z);
    const bool on_plane = ap.axis >= 0 && coord == ap.plane;
    const T kPi = ap.consistent ? (T)1.5 : (T)-0.5;
    const T lPit = lPis;
    const T lCu = kPi * lPis;
    T lJ[3], lCv[3], luav[3];
    T ln = lns + lntot;
    T dot = 0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        lCv[c] = lCs[c] + ua[c] * lCu;
        luav[c] = lua[c] + Cv[c] * lCu;
        lJ[c] = lJtot[c] + luav[c] * inv_n;
        dot += luav[c] * ua[c];
    }
    ln -= dot * inv_n;
    if (on_plane) lJ[ap.axis] += (T)ap.wobj;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const T lnF = lnFs[c] + (T)0.5 * lJ[c];
        if (!ap.consistent) lCv[c] += (T)0.5 * lJ[c];
        ln += lnF * Fv[c];
        lF[((long long)a * 3 + c) * g.N + i] += n * lnF;
        lC[((long long)a * 3 + c) * g.N + i] = lCv[c];
    }
    const T om1 = (T)1 - om;
    [&]<int... P>(std::integer_sequence<int, P...>) {
        (
            [&] {
                of[(long long)P * g.N] = om1 * lf[P] + ln;
                if constexpr (P == 0)
                    og[0] = om1 * lg[0] + lPit;
                else
                    og[(long long)P * g.N] = om1 * lg[P] + lPit + link_dot<T, P>(lJ);
            }(),
            ...);
    }(std::make_integer_sequence<int, Q>{});
}

cudaError_t launch_adj_collide_pair(Prec p, const Grid &g, const void *post, const uint32_t *mask, const void *C,
                                   const void *F, const AdjParams &ap, const void *lYf_in, const void *lYg_in,
                                   const void *lnd_in, void *lYf_out, void *lYg_out, void *lC, void *lF,
                                   cudaStream_t st) {
    const int per_cta = ap.M == 2 ? ACP / 2 : ACP;
    const unsigned nb = (unsigned)((g.N + per_cta - 1) / per_cta);
#define LBE_ADJ_PAIR(SS, TT, MM)                                                                                \
    k_adj_collide_pair<SS, TT, MM><<<nb, ACP, 0, st>>>(g, (const SS *)post, mask, (const TT *)C, (const TT *)F, \
                                                       ap, (const TT *)lYf_in, (const TT *)lYg_in,               \
                                                       (const TT *)lnd_in, (TT *)lYf_out, (TT *)lYg_out,         \
                                                       (TT *)lC, (TT *)lF)
    if (p == Prec::F64) {
        if (ap.M == 1) LBE_ADJ_PAIR(double, double, 1); else LBE_ADJ_PAIR(double, double, 2);
    } else if (p == Prec::F32) {
        if (ap.M == 1) LBE_ADJ_PAIR(float, float, 1); else LBE_ADJ_PAIR(float, float, 2);
    } else {
        return cudaErrorInvalidValue;
    }
#undef LBE_ADJ_PAIR
    return cudaGetLastError();
}

}  // namespace lbe
