// K4: fused moments + DD-TR collision + pull streaming (Sec. "Hard sphere fluid mixture in a potential well"; the
// collision itself is in lbe_collide.cuh), and K1 for one species.
//
// Two species or more: a CTA takes 128 consecutive nodes (fewer on small lattices), warps 4a .. 4a + 3 species a of
// the same nodes, 32 consecutive nodes per warp.  Each thread pulls only its own species' 38 populations, keeps them
// in registers, computes that species' moments, and gets the other species' n and J through shared memory to form the
// barycentric velocity u = sum J / sum n.  A warp's load of one population is one 128-byte run of one species'
// array (FP32), as in the one-species kernel.  Compared with one thread per node holding every species, the live
// state per thread shrinks to one species', so more warps share an SM, and nothing is pulled twice.
// One species: one thread per node, 32 consecutive nodes per warp, u = J/n.
//
// Bounds: HBM with FP32 storage (785 us for the 512x128x128 channel's 5.1 GB, 96% of the measured copy bandwidth; 886
// before the collision's pairs shared their parts); the FP64 pipe in FP64 (256x64x64 channel 2.55 -> 0.81 ms: 1.20
// with shared pairs and two CTAs, 0.99 with the moments on the integer pipe, the rest by Collision64); issue with 16-bit storage
// (channel 887 -> 695 us, half of them integer instructions for addresses and conversions).  Three species: the
// kernel with one thread per node for all of them pulled every population twice (90x75x66 166 -> 86 us).
#include <math.h>

#include <type_traits>
#include <utility>

#include "lbe_collide.cuh"
#include "lbe_device.cuh"
#include "lbe_launch.h"
#include "lbe_node.cuh"

namespace lbe {

constexpr int NTP = 256;  // threads per CTA of one species (256 nodes)
constexpr int NPC = 128;  // nodes per CTA of a mixture (one group of 128 threads per species)
__host__ __device__ constexpr int collide_threads(int M) { return M == 1 ? NTP : M * NPC; }
// CTAs per SM the registers are held to, the fastest of those measured (K4 of the 256^3 well, FP32: two 1.01 ms,
// three 0.815, four 0.834; 512x128x128 channel, FP32: two 0.92, three 0.82, four 0.96; BF16: two 0.90, three 0.72,
// four 0.74; 256x64x64 channel, FP64: one 1.33, two 1.20, three 1.21).
__host__ __device__ constexpr int collide_ctas(int M, bool f32) {
    return !f32 ? (M <= 2 ? 2 : 1) : (M <= 2 ? 3 : (M == 3 ? 2 : 1));
}

template <typename S, typename T, int M, bool SOLID>
__global__ void __launch_bounds__(collide_threads(M), collide_ctas(M, sizeof(T) == 4))
    k_collide_pair(Grid g, const S *__restrict__ src, S *__restrict__ dst, const uint32_t *__restrict__ mask,
                   const T *__restrict__ C, const T *__restrict__ F, StepParams sp, double *__restrict__ flux_buf,
                   int lg) {
    pdl_wait();
    const int a = M >= 2 ? (int)(threadIdx.x >> lg) : 0;           // species of this thread
    const int loc = M >= 2 ? (int)(threadIdx.x & ((1 << lg) - 1)) : 0;  // node within the CTA's 2^lg (128 at most)
    const long long i = M >= 2 ? ((long long)blockIdx.x << lg) + loc : (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = i < g.N;
    int x = 0, y = 0, z = 0;
    if (valid) node_xyz(g, i, x, y, z);
    const uint32_t m = valid ? (SOLID ? mask[i] : 0u) : 1u;
    const bool fluid = !(m & 1u);
    const int coord = sp.flux_axis == 0 ? x : (sp.flux_axis == 1 ? y : z);
    const bool on_plane = valid && sp.flux_axis >= 0 && coord == sp.flux_plane;
    const int psize = sp.flux_axis == 0 ? g.ny * g.nz : (sp.flux_axis == 1 ? g.nx * g.nz : g.nx * g.ny);

    // this species' constants (selected, not indexed, so the parameter block stays in constant memory)
    // (16-bit storage takes the float copies rounded on the host; the doubles are then unused)
    const SpeciesConst &sc = M == 1 ? sp.sp[0] : (M == 2 ? (a == 0 ? sp.sp[0] : sp.sp[1]) : sp.sp[a]);
    // a warp none of whose nodes has a blocked link pulls without the bounce-back selects
    const bool plain = !SOLID || __all_sync(0xffffffffu, (m >> 1) == 0u);
    // moments of this thread's species (zero on solid nodes and past the end)
    // FP32 storage, three or four species: on f itself, population by population, which is the rounding such runs
    // have always had (the deviations round less, 5.7e-7 against 4.5e-6 of the velocity after 20 steps of a ternary
    // well, but shift a run by that difference)
    constexpr bool WHOLE = M >= 3 && std::is_same_v<S, float>;
    constexpr bool DEV = Store<S, T>::shifted && !WHOLE, UNIT = sizeof(S) == 2;
    T f[Q], gq[Q];
    T n = 0, dn = 0, Pi = 0, J[3] = {0, 0, 0}, Cv[3] = {0, 0, 0}, nF[3] = {0, 0, 0}, ua[3] = {0, 0, 0};
    if (fluid) {
        const NbrOff o = nbr_offsets(g, x, y, z);
        // mixtures: C and F issue with the populations, so their latency is not paid again after the moment sums
        // (512x128x128 channel, FP32 0.99 -> 0.90 ms when it was made, BF16 0.77 -> 0.72); for one species the
        // early loads measured slower (256^3 well 0.834 -> 0.879): they stay after the sums there
        constexpr bool CF_EARLY = M >= 2;
        T Fv[3];
        if constexpr (CF_EARLY) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                Cv[c] = C[((long long)a * 3 + c) * g.N + i];
                Fv[c] = F[((long long)a * 3 + c) * g.N + i];
            }
        }
        const T n0 = sc_n0<S, T>(sc);
        const S *fb = src + pop_off(a, 0, 0, g.N);
        const S *gb = src + pop_off(a, 1, 0, g.N);
        auto take = [&](auto Pc, auto Sc) {
            constexpr int P = decltype(Pc)::value;
            constexpr bool SEL = decltype(Sc)::value;
            if constexpr (WHOLE) {
                f[P] = pull<S, T, P, SEL>(fb, g.N, i, o, m, n0);
            } else {
                f[P] = pull_unit<S, T, P, SEL>(fb, g.N, i, o, m);
            }
        };
        auto takeg = [&](auto Pc, auto Sc) {
            constexpr int P = decltype(Pc)::value;
            constexpr bool SEL = decltype(Sc)::value;
            if constexpr (WHOLE) {
                gq[P] = pull<S, T, P, SEL>(gb, g.N, i, o, m, n0);
            } else {
                gq[P] = pull_unit<S, T, P, SEL>(gb, g.N, i, o, m);
            }
        };
        // one branch for both distributions: all 38 loads issue together (two branches: 0.89 instead of 0.82 ms, FP32)
        if (plain) {
            [&]<int... P>(std::integer_sequence<int, P...>) {
                (take(std::integral_constant<int, P>{}, std::false_type{}), ...);
                (takeg(std::integral_constant<int, P>{}, std::false_type{}), ...);
            }(std::make_integer_sequence<int, Q>{});
        } else {
            [&]<int... P>(std::integer_sequence<int, P...>) {
                (take(std::integral_constant<int, P>{}, std::bool_constant<SOLID>{}), ...);
                (takeg(std::integral_constant<int, P>{}, std::bool_constant<SOLID>{}), ...);
            }(std::make_integer_sequence<int, Q>{});
        }
        // n and Pi~ (DEV: their deviations from n0; the rest values sum to n0, and to zero in J~)
        T Pit, Jt[3];
        n = zeroth_moment<UNIT>(f);
        if constexpr (WHOLE) {
            Pit = zeroth_moment<false>(gq);
            ordered_momentum(gq, Jt);
        } else {
            pair_moments<UNIT>(gq, Pit, Jt);
        }
        if constexpr (UNIT) {
            const T s = (T)(1.0 / 36.0) * n0;
            n *= s;
            Pit *= s;
#pragma unroll
            for (int c = 0; c < 3; ++c) Jt[c] *= s;
        }
        if constexpr (DEV) {
            dn = n;
            n = n0 + dn;
        }
        const T inv_n = n > (T)0 ? (T)1 / n : (T)0;
        T Cu = 0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if constexpr (!CF_EARLY) {
                Cv[c] = C[((long long)a * 3 + c) * g.N + i];
                Fv[c] = F[((long long)a * 3 + c) * g.N + i];
            }
            nF[c] = n * Fv[c];
            J[c] = sp.consistent ? Jt[c] + (T)0.5 * nF[c] : Jt[c] + (T)0.5 * (Cv[c] + nF[c]);
            ua[c] = J[c] * inv_n;
            Cu += Cv[c] * ua[c];
        }
        Pi = sp.consistent ? Pit + (T)1.5 * Cu : Pit - (T)0.5 * Cu;  // DEV: Pi - n0
    }
    // the other species of the same node, through shared memory; every thread takes part
    T ntot = n, Jtot[3] = {J[0], J[1], J[2]};
    if constexpr (M >= 2) {
        __shared__ T xch[M][4][NPC];
        xch[a][0][loc] = n;
#pragma unroll
        for (int c = 0; c < 3; ++c) xch[a][c + 1][loc] = J[c];
        // only the M warps over the same 32 nodes (one of each species) wait for each other: named barrier 1 + w of
        // 32 M threads (barrier 0 is the block's); 0.897 -> 0.885 ms on the 512x128x128 channel against the block
        // barrier
        asm volatile("bar.sync %0, %1;" ::"r"(1 + (loc >> 5)), "n"(32 * M) : "memory");
        ntot = xch[0][0][loc];
#pragma unroll
        for (int c = 0; c < 3; ++c) Jtot[c] = xch[0][c + 1][loc];
#pragma unroll
        for (int b = 1; b < M; ++b) {
            ntot += xch[b][0][loc];
#pragma unroll
            for (int c = 0; c < 3; ++c) Jtot[c] += xch[b][c + 1][loc];
        }
    }
    if (on_plane)
        flux_buf[(long long)a * psize + plane_index(g, sp.flux_axis, x, y, z)] =
            fluid ? (double)J[sp.flux_axis] : 0.0;
    if (!fluid) return;
    const T inv_tot = ntot > (T)0 ? (T)1 / ntot : (T)0;
    T u[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) u[c] = Jtot[c] * inv_tot;
    S *fo = dst + pop_off(a, 0, 0, g.N) + i;
    S *go = dst + pop_off(a, 1, 0, g.N) + i;
    auto put = [&](auto Pc, T fs, T gs) {
        constexpr int P = decltype(Pc)::value;
        Store<S, T>::store_unit(fo + (long long)P * g.N, fs);
        Store<S, T>::store_unit(go + (long long)P * g.N, gs);
    };
    if constexpr (WHOLE) {
        collide_whole(n, Pi, ua, u, Cv, nF, (T)sc.omega_eff, (T)sc.inv, f, gq);
        const T n0s = sc_n0<S, T>(sc);
        [&]<int... P>(std::integer_sequence<int, P...>) {
            (put(std::integral_constant<int, P>{}, f[P] - (T)wq(P) * n0s, gq[P] - (T)wq(P) * n0s), ...);
        }(std::make_integer_sequence<int, Q>{});
        return;
    }
    if constexpr (sizeof(T) == 8) {
        Collision64 col;
        col.set(n, Pi, ua, u, Cv, nF, sc.omega_eff, sc.inv);
        auto half = [&](S *out, T(&v)[Q]) {
            col.rest(v[0]);
            Store<S, T>::store_unit(out, v[0]);
            [&]<int... K>(std::integer_sequence<int, K...>) {
                (
                    [&] {
                        constexpr int P = 2 * K + 1;
                        col.template pair<P>(v[P], v[P + 1]);
                        Store<S, T>::store_unit(out + (long long)P * g.N, v[P]);
                        Store<S, T>::store_unit(out + (long long)(P + 1) * g.N, v[P + 1]);
                    }(),
                    ...);
            }(std::make_integer_sequence<int, 9>{});
        };
        half(fo, f);
        col.next();
        half(go, gq);
        return;
    }
    Collision<T, UNIT> col;
    col.set(n, DEV ? dn : n, Pi, J, ua, u, Cv, nF, sc_omega<S, T>(sc), sc_inv<S, T>(sc),
            UNIT ? sc_in0<S, T>(sc) : (T)0);
    col.rest(f[0], gq[0]);
    put(std::integral_constant<int, 0>{}, f[0], gq[0]);
    [&]<int... K>(std::integer_sequence<int, K...>) {
        (
            [&] {
                constexpr int P = 2 * K + 1;
                col.template pair<P>(f[P], f[P + 1], gq[P], gq[P + 1]);
                put(std::integral_constant<int, P>{}, f[P], gq[P]);
                put(std::integral_constant<int, P + 1>{}, f[P + 1], gq[P + 1]);
            }(),
            ...);
    }(std::make_integer_sequence<int, 9>{});
}

// K1 for one species: n(r) = sum_p f~_p(r) pulled, 0 on solid nodes, into the padded stencil field with its
// periodic images (the arithmetic of k_density).
template <typename S, typename T, bool SOLID>
__global__ void __launch_bounds__(NTP)
    k_density_pair(Grid g, const S *__restrict__ pop, const uint32_t *__restrict__ mask, double n00,
                   T *__restrict__ npad, int *err) {
    pdl_wait();
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = i < g.N;
    const uint32_t m = valid ? (SOLID ? mask[i] : 0u) : 1u;
    // a warp none of whose nodes has a blocked link pulls without the bounce-back selects
    const bool plain = !SOLID || __all_sync(0xffffffffu, (m >> 1) == 0u);
    if (!valid) return;
    int x, y, z;
    node_xyz(g, i, x, y, z);
    T n = (T)0;
    if (!(m & 1u)) {
        const NbrOff o = nbr_offsets(g, x, y, z);
        T v[Q];
        pull_all<S, T, SOLID>(pop, g.N, i, o, m, plain, v);
        n = density_of<S, T>(v, (T)n00);
        if (!(n >= (T)0) || !isfinite(n)) atomicOr(err, ERR_DENSITY);
    }
    write_padded<T>(g, npad, x, y, z, n);
}

#define LBE_PAIR_DISPATCH(p, ...)                                                      \
    switch (p) {                                                                       \
        case Prec::F64: { using S = double; using T = double; __VA_ARGS__; break; }    \
        case Prec::F32: { using S = float; using T = float; __VA_ARGS__; break; }      \
        case Prec::BF16: { using S = __nv_bfloat16; using T = float; __VA_ARGS__; break; } \
        case Prec::F16: { using S = __half; using T = float; __VA_ARGS__; break; }     \
    }

cudaError_t launch_collide(Prec p, const Grid &g, const void *src, void *dst, const uint32_t *mask, bool solid,
                           const void *C, const void *F, const StepParams &sp, double *flux_buf, cudaStream_t st) {
    // nodes per CTA: 256 (one species) or 128, fewer on small lattices (24^3, FP64: 30.4 -> 18.3 us)
    int lg = 7;
    while (sp.M >= 2 && lg > 5 && ((g.N + (1 << lg) - 1) >> lg) < 2 * 152) --lg;
    const int per_cta = sp.M >= 2 ? 1 << lg : node_threads(g.N, NTP);
    const int threads = sp.M >= 2 ? sp.M << lg : per_cta;
    const unsigned nb = (unsigned)((g.N + per_cta - 1) / per_cta);
    cudaError_t e = cudaSuccess;
#define LBE_PAIR(MM, SOL)                                                                                       \
    e = launch_pdl(k_collide_pair<S, T, MM, SOL>, nb, threads, 0, st, g, (const S *)src, (S *)dst, mask,        \
                   (const T *)C, (const T *)F, sp, flux_buf, lg)
#define LBE_PAIR_M(MM)                          \
    if (solid) {                                \
        LBE_PAIR_DISPATCH(p, LBE_PAIR(MM, true)); \
    } else {                                    \
        LBE_PAIR_DISPATCH(p, LBE_PAIR(MM, false)); \
    }
    switch (sp.M) {
        case 1: LBE_PAIR_M(1) break;
        case 2: LBE_PAIR_M(2) break;
        case 3: LBE_PAIR_M(3) break;
        case 4: LBE_PAIR_M(4) break;
        default: return cudaErrorInvalidValue;
    }
#undef LBE_PAIR_M
#undef LBE_PAIR
    return e;
}

cudaError_t launch_density_pair(Prec p, const Grid &g, const void *pop, const uint32_t *mask, bool solid,
                                double n0, void *npad, int *err, cudaStream_t st) {
    const int threads = node_threads(g.N, NTP);
    const unsigned nb = (unsigned)((g.N + threads - 1) / threads);
    cudaError_t e = cudaSuccess;
#define LBE_DPAIR(SOL) \
    e = launch_pdl(k_density_pair<S, T, SOL>, nb, threads, 0, st, g, (const S *)pop, mask, n0, (T *)npad, err)
    if (solid) {
        LBE_PAIR_DISPATCH(p, LBE_DPAIR(true));
    } else {
        LBE_PAIR_DISPATCH(p, LBE_DPAIR(false));
    }
#undef LBE_DPAIR
    return e;
}

}  // namespace lbe
