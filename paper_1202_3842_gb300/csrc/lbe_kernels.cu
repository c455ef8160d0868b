// D3Q19 Lattice Boltzmann-Enskog kernels (sm_103a): geometry, force field,
// population set/get, K1 density, moments and FP64 reductions.  The contact values (K2) are in lbe_contact.cuh,
// the shell force (K3) in lbe_shell_march.cuh and lbe_shell_fixed.cuh, the collision (K4) in lbe_collide_pair.cu.
//
// Population storage: [M][2 (f, g)][19][N] of the storage type S, holding the
// post-collision populations f~*(r, t-1); the streamed populations of step t
// are pulled: f~_p(r, t) = f~*_p(r - c_p, t-1), or f~*_{opp(p)}(r, t-1) when
// the link is blocked (mid-point bounce-back, Sec. "Channel flow with a
// bottleneck").  Link mask bit 0 marks a solid node, bit p a blocked link p.
#include <math.h>

#include <utility>

#include "lbe_collide.cuh"
#include "lbe_device.cuh"
#include "lbe_launch.h"
#include "lbe_node.cuh"

namespace lbe {

constexpr int NT = 256;

struct N0Vec {
    double v[MAXS];
};
struct N0VecF {  // the same rounded once on the host, read with 16-bit storage
    float v[MAXS];
};

// ---------------------------------------------------------------------------
// geometry
// ---------------------------------------------------------------------------
__global__ void k_link_mask(Grid g, const uint8_t *__restrict__ solid, uint32_t *__restrict__ mask) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.N) return;
    int x, y, z;
    node_xyz(g, i, x, y, z);
    uint32_t m = solid[i] ? 1u : 0u;
#pragma unroll
    for (int p = 1; p < Q; ++p) {
        int X = x - cx(p), Y = y - cy(p), Z = z - cz(p);
        bool ok = wrap(X, g.nx, g.per[0]) && wrap(Y, g.ny, g.per[1]) && wrap(Z, g.nz, g.per[2]);
        if (!ok || solid[X + (long long)g.nx * (Y + (long long)g.ny * Z)]) m |= (1u << p);
    }
    mask[i] = m;
}

cudaError_t launch_link_mask(const Grid &g, const uint8_t *solid, uint32_t *mask, cudaStream_t st) {
    k_link_mask<<<(unsigned)((g.N + NT - 1) / NT), NT, 0, st>>>(g, solid, mask);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// force field F = -grad_h V + g  (isotropic D3Q19 gradient, FP64 arithmetic)
// ---------------------------------------------------------------------------
template <typename T>
__global__ void k_force_field(Grid g, const double *__restrict__ V, const double *__restrict__ phi,
                              const double *__restrict__ amp, double g0, double g1, double g2, T *__restrict__ F) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.N) return;
    int x, y, z;
    node_xyz(g, i, x, y, z);
    const double vi = V[i] + amp[i] * phi[i];
    double gr[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int p = 1; p < Q; ++p) {
        int X = x + cx(p), Y = y + cy(p), Z = z + cz(p);
        bool ok = wrap(X, g.nx, g.per[0]) && wrap(Y, g.ny, g.per[1]) && wrap(Z, g.nz, g.per[2]);
        double v = vi;
        if (ok) {
            long long j = X + (long long)g.nx * (Y + (long long)g.ny * Z);
            v = V[j] + amp[j] * phi[j];
        }
        gr[0] += wq(p) * cx(p) * v;
        gr[1] += wq(p) * cy(p) * v;
        gr[2] += wq(p) * cz(p) * v;
    }
    F[i] = (T)(-3.0 * gr[0] + g0);
    F[g.N + i] = (T)(-3.0 * gr[1] + g1);
    F[2 * g.N + i] = (T)(-3.0 * gr[2] + g2);
}

cudaError_t launch_force_field(Prec p, const Grid &g, const double *V, const double *phi, const double *amp,
                               const double gb[3], void *F, cudaStream_t st) {
    unsigned nb = (unsigned)((g.N + NT - 1) / NT);
    if (prec_fp64(p))
        k_force_field<double><<<nb, NT, 0, st>>>(g, V, phi, amp, gb[0], gb[1], gb[2], (double *)F);
    else
        k_force_field<float><<<nb, NT, 0, st>>>(g, V, phi, amp, gb[0], gb[1], gb[2], (float *)F);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// populations: streamed FP64 <-> stored post-collision form
// ---------------------------------------------------------------------------
// post_p(s) = streamed_p(s + c_p) when s + c_p is a fluid node inside the
// lattice, else streamed_{opp(p)}(s) (the population bounced back at s).
// A population given in FP64 (host data, rest state) stored in the storage form: the shifted forms take
// the deviation f - w_p n0 formed in FP64, so it keeps its precision.
template <typename S, typename T>
__device__ __forceinline__ void store_full(S *p, double v, double wn0) {
    if constexpr (Store<S, T>::shifted)
        Store<S, T>::store_dev(p, (T)(v - wn0), (T)wn0, wn0 > 0.0 ? (T)(1.0 / wn0) : (T)0);
    else
        Store<S, T>::store(p, (T)v, (T)wn0, (T)0);
}

// The FP64 value of a stored population (the shifted forms add w_p n0 in FP64).
template <typename S, typename T, int P>
__device__ __forceinline__ double pull_full(const S *fb, long long N, long long i, const NbrOff &o, uint32_t m,
                                            double n0) {
    if constexpr (Store<S, T>::shifted)
        return (double)pull_dev<S, T, P>(fb, N, i, o, m, (T)n0) + wq(P) * n0;
    else
        return (double)pull<S, T, P>(fb, N, i, o, m, (T)n0);
}

template <typename S, typename T>
__global__ void k_unstream(Grid g, const uint32_t *__restrict__ mask, const double *__restrict__ f,
                           const double *__restrict__ gq, S *__restrict__ pop, int a, double n0) {
    long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= g.N) return;
    int x, y, z;
    node_xyz(g, s, x, y, z);
    const bool solid = mask[s] & 1u;
#pragma unroll
    for (int p = 0; p < Q; ++p) {
        double fv = 0.0, gv = 0.0;
        if (!solid) {
            int X = x + cx(p), Y = y + cy(p), Z = z + cz(p);
            bool ok = wrap(X, g.nx, g.per[0]) && wrap(Y, g.ny, g.per[1]) && wrap(Z, g.nz, g.per[2]);
            long long t = ok ? X + (long long)g.nx * (Y + (long long)g.ny * Z) : 0;
            if (ok && !(mask[t] & 1u)) {
                fv = f[(long long)p * g.N + t];
                gv = gq[(long long)p * g.N + t];
            } else {
                fv = f[(long long)opp(p) * g.N + s];
                gv = gq[(long long)opp(p) * g.N + s];
            }
        }
        store_full<S, T>(pop + pop_off(a, 0, p, g.N) + s, fv, wq(p) * n0);
        store_full<S, T>(pop + pop_off(a, 1, p, g.N) + s, gv, wq(p) * n0);
    }
}

// Rest state: streamed f_p(r) = w_p n(r) and g_p(r) = w_p Pi(r) on fluid nodes (Pi = n without pi).
template <typename S, typename T>
__global__ void k_rest_state(Grid g, const uint32_t *__restrict__ mask, const double *__restrict__ n,
                             const double *__restrict__ pi, S *__restrict__ pop, int a, double n0) {
    long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= g.N) return;
    int x, y, z;
    node_xyz(g, s, x, y, z);
    const bool solid = mask[s] & 1u;
    const double *gsrc = pi ? pi : n;
#pragma unroll
    for (int p = 0; p < Q; ++p) {
        double v = 0.0, vg = 0.0;
        if (!solid) {
            int X = x + cx(p), Y = y + cy(p), Z = z + cz(p);
            bool ok = wrap(X, g.nx, g.per[0]) && wrap(Y, g.ny, g.per[1]) && wrap(Z, g.nz, g.per[2]);
            long long t = ok ? X + (long long)g.nx * (Y + (long long)g.ny * Z) : 0;
            const long long u = (ok && !(mask[t] & 1u)) ? t : s;
            v = wq(p) * n[u];
            vg = wq(p) * gsrc[u];
        }
        store_full<S, T>(pop + pop_off(a, 0, p, g.N) + s, v, wq(p) * n0);
        store_full<S, T>(pop + pop_off(a, 1, p, g.N) + s, vg, wq(p) * n0);
    }
}

template <typename S, typename T>
__global__ void k_stream_out(Grid g, const uint32_t *__restrict__ mask, const S *__restrict__ pop, int a, double n0,
                             double *__restrict__ f, double *__restrict__ gq) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.N) return;
    int x, y, z;
    node_xyz(g, i, x, y, z);
    const uint32_t m = mask[i];
    const NbrOff o = nbr_offsets(g, x, y, z);
    const S *fb = pop + pop_off(a, 0, 0, g.N);
    const S *gb = pop + pop_off(a, 1, 0, g.N);
    auto body = [&](auto Pc) {
        constexpr int P = decltype(Pc)::value;
        double fv = 0.0, gv = 0.0;
        if (!(m & 1u)) {
            fv = pull_full<S, T, P>(fb, g.N, i, o, m, n0);
            gv = pull_full<S, T, P>(gb, g.N, i, o, m, n0);
        }
        f[(long long)P * g.N + i] = fv;
        gq[(long long)P * g.N + i] = gv;
    };
    [&]<int... P>(std::integer_sequence<int, P...>) { (body(std::integral_constant<int, P>{}), ...); }
    (std::make_integer_sequence<int, Q>{});
}

#define LBE_DISPATCH_PREC(p, CALL)                                       \
    switch (p) {                                                         \
        case Prec::F64: { using S = double; using T = double; CALL; break; }      \
        case Prec::F32: { using S = float; using T = float; CALL; break; }        \
        case Prec::BF16: { using S = __nv_bfloat16; using T = float; CALL; break; } \
        case Prec::F16: { using S = __half; using T = float; CALL; break; }       \
    }

cudaError_t launch_unstream(Prec p, const Grid &g, const uint32_t *mask, const double *f, const double *gq,
                            void *pop, int a, double n0, cudaStream_t st) {
    unsigned nb = (unsigned)((g.N + NT - 1) / NT);
    LBE_DISPATCH_PREC(p, (k_unstream<S, T><<<nb, NT, 0, st>>>(g, mask, f, gq, (S *)pop, a, n0)));
    return cudaGetLastError();
}

cudaError_t launch_rest_state(Prec p, const Grid &g, const uint32_t *mask, const double *n, void *pop, int a,
                              double n0, cudaStream_t st, const double *pi) {
    unsigned nb = (unsigned)((g.N + NT - 1) / NT);
    LBE_DISPATCH_PREC(p, (k_rest_state<S, T><<<nb, NT, 0, st>>>(g, mask, n, pi, (S *)pop, a, n0)));
    return cudaGetLastError();
}

cudaError_t launch_stream_out(Prec p, const Grid &g, const uint32_t *mask, const void *pop, int a, double n0,
                              double *f, double *gq, cudaStream_t st) {
    unsigned nb = (unsigned)((g.N + NT - 1) / NT);
    LBE_DISPATCH_PREC(p, (k_stream_out<S, T><<<nb, NT, 0, st>>>(g, mask, (const S *)pop, a, n0, f, gq)));
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// K1: density n^a(r) = sum_p f~_p(r) (streamed), 0 on solid nodes, written to
// the padded stencil field with its periodic images.
// ---------------------------------------------------------------------------
template <typename S, typename T, bool SOLID, int MC>
__global__ void __launch_bounds__(NT) k_density(Grid g, const S *__restrict__ pop, const uint32_t *__restrict__ mask,
                                                N0Vec n0v, N0VecF n0f, T *__restrict__ npad, int *err) {
    pdl_wait();
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = i < g.N;
    const uint32_t m = valid ? (SOLID ? mask[i] : 0u) : 1u;
    // a warp none of whose nodes has a blocked link pulls without the bounce-back selects
    // (0.257 -> 0.227 ms on the 512x128x128 channel)
    const bool plain = (!SOLID || __all_sync(0xffffffffu, (m >> 1) == 0u));
    if (!valid) return;
    int x, y, z;
    node_xyz(g, i, x, y, z);
    const NbrOff o = nbr_offsets(g, x, y, z);  // (without solids every axis is periodic)
    auto n0_of = [&](int a) -> T {
        if constexpr (sc_float<S, T>)
            return n0f.v[a];
        else
            return (T)n0v.v[a];
    };
    auto pull_species = [&](int a, T(&v)[Q]) {
        pull_all<S, T, SOLID>(pop + pop_off(a, 0, 0, g.N), g.N, i, o, m, plain, v);
    };
    auto finish = [&](int a, const T *v) -> T {
        const T n = density_of<S, T>(v, n0_of(a));
        if (!(n >= (T)0) || !isfinite(n)) atomicOr(err, ERR_DENSITY);
        return n;
    };
    T n[MC];
#pragma unroll
    for (int a = 0; a < MC; ++a) n[a] = (T)0;
    if (!(m & 1u)) {
        if constexpr (MC == 2) {  // all 38 loads issue before either sum
            T v0[Q], v1[Q];
            pull_species(0, v0);
            pull_species(1, v1);
            n[0] = finish(0, v0);
            n[1] = finish(1, v1);
        } else {
#pragma unroll
            for (int a = 0; a < MC; ++a) {
                T v[Q];
                pull_species(a, v);
                n[a] = finish(a, v);
            }
        }
    }
#pragma unroll
    for (int a = 0; a < MC; ++a) write_padded<T>(g, npad + (long long)a * g.P, x, y, z, n[a]);
}

cudaError_t launch_density(Prec p, const Grid &g, const void *pop, const uint32_t *mask, bool solid, int M,
                           const double *n0, void *npad, int *err, cudaStream_t st) {
    // one species: one thread per node at 32-42 registers (lbe_collide_pair.cu); measured faster than this
    // kernel for one species (256^3 well 0.42 -> 0.31 ms) and slower for two (0.29 -> 0.31 ms)
    if (M == 1) return launch_density_pair(p, g, pop, mask, solid, n0[0], npad, err, st);
    const int threads = node_threads(g.N, NT);
    const unsigned nb = (unsigned)((g.N + threads - 1) / threads);
    N0Vec n0v;
    N0VecF n0f;
    for (int a = 0; a < MAXS; ++a) {
        n0v.v[a] = a < M ? n0[a] : 0.0;
        n0f.v[a] = (float)n0v.v[a];
    }
    cudaError_t e = cudaSuccess;
#define LBE_K1(SOL, MC) \
    LBE_DISPATCH_PREC(p, (e = launch_pdl(k_density<S, T, SOL, MC>, nb, threads, 0, st, g, (const S *)pop, mask, n0v, n0f, (T *)npad, err)))
#define LBE_K1_M(MC)       \
    if (solid) {           \
        LBE_K1(true, MC);  \
    } else {               \
        LBE_K1(false, MC); \
    }
    switch (M) {
        case 2: LBE_K1_M(2) break;
        case 3: LBE_K1_M(3) break;
        case 4: LBE_K1_M(4) break;
        default: return cudaErrorInvalidValue;
    }
#undef LBE_K1_M
#undef LBE_K1
    return e;
}

// ---------------------------------------------------------------------------
// Moments of the current state (the collision itself: lbe_collide_pair.cu):
//   n = sum f~, Pi~ = sum g~, J~ = sum c g~;
//   printed recovery:    J = J~ + (C + nF)/2;
//   consistent recovery: J = J~ + nF/2.
// ---------------------------------------------------------------------------
// For the getters: n [M][N], J [M][3][N] (FP64).
template <typename S, typename T, int M>
__global__ void __launch_bounds__(NT) k_moments(Grid g, const S *__restrict__ src, const uint32_t *__restrict__ mask,
                                                const T *__restrict__ C, const T *__restrict__ F, StepParams sp,
                                                double *__restrict__ nout, double *__restrict__ Jout) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.N) return;
    int x, y, z;
    node_xyz(g, i, x, y, z);
    const uint32_t m = mask[i];
    const bool solid = m & 1u;
    NbrOff o{};
    if (!solid) o = nbr_offsets(g, x, y, z);
#pragma unroll
    for (int a = 0; a < M; ++a) {
        T n = 0, J[3] = {0, 0, 0};
        if (!solid) {
            const T n0 = sc_n0<S, T>(sp.sp[a]);
            const S *fb = src + pop_off(a, 0, 0, g.N);
            const S *gb = src + pop_off(a, 1, 0, g.N);
            T f[Q], gq[Q], Pi;
            [&]<int... P>(std::integer_sequence<int, P...>) {
                ((f[P] = pull<S, T, P, true>(fb, g.N, i, o, m, n0)), ...);
                ((gq[P] = pull<S, T, P, true>(gb, g.N, i, o, m, n0)), ...);
            }(std::make_integer_sequence<int, Q>{});
            n = zeroth_moment<false>(f);
            if constexpr (sizeof(T) == 4)  // rounds as the getters always have
                ordered_momentum(gq, J);
            else
                pair_moments<false>(gq, Pi, J);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const T Cc = C[((long long)a * 3 + c) * g.N + i];
                const T nF = n * F[((long long)a * 3 + c) * g.N + i];
                J[c] += (T)0.5 * (sp.consistent ? nF : Cc + nF);
            }
        }
        nout[(long long)a * g.N + i] = (double)n;
#pragma unroll
        for (int c = 0; c < 3; ++c) Jout[((long long)a * 3 + c) * g.N + i] = (double)J[c];
    }
}

template <typename S, typename T>
static cudaError_t moments_m(int M, const Grid &g, const void *pop, const uint32_t *mask, const void *C, const void *F,
                             const StepParams &sp, double *n, double *J, cudaStream_t st) {
    const int nt = node_threads(g.N, NT);
    const unsigned nb = (unsigned)((g.N + nt - 1) / nt);
    switch (M) {
        case 1: k_moments<S, T, 1><<<nb, nt, 0, st>>>(g, (const S *)pop, mask, (const T *)C, (const T *)F, sp, n, J); break;
        case 2: k_moments<S, T, 2><<<nb, nt, 0, st>>>(g, (const S *)pop, mask, (const T *)C, (const T *)F, sp, n, J); break;
        case 3: k_moments<S, T, 3><<<nb, nt, 0, st>>>(g, (const S *)pop, mask, (const T *)C, (const T *)F, sp, n, J); break;
        case 4: k_moments<S, T, 4><<<nb, nt, 0, st>>>(g, (const S *)pop, mask, (const T *)C, (const T *)F, sp, n, J); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_moments(Prec p, const Grid &g, const void *pop, const uint32_t *mask, const void *C,
                           const void *F, const StepParams &sp, double *n, double *J, cudaStream_t st) {
    cudaError_t e = cudaSuccess;
    LBE_DISPATCH_PREC(p, (e = moments_m<S, T>(sp.M, g, pop, mask, C, F, sp, n, J, st)));
    return e;
}

// ---------------------------------------------------------------------------
// K5 and FP64 reductions (deterministic: fixed per-thread order, fixed tree).
// ---------------------------------------------------------------------------
template <int NTH>
__device__ __forceinline__ double block_sum(double v, double *sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    if (wid == 0) {
        v = lane < NTH / 32 ? sh[lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    }
    __syncthreads();
    return v;  // valid in thread 0
}
template <int NTH>
__device__ __forceinline__ double block_max(double v, double *sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    if (wid == 0) {
        v = lane < NTH / 32 ? sh[lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    }
    __syncthreads();
    return v;
}

// One block per species; four partial sums per thread, so that four loads are in flight (one block for all species
// and one load at a time: 20 us for two 128 x 128 planes, 13.6 now, with the events around it).
__global__ void __launch_bounds__(1024) k_flux_reduce(int psize, const double *__restrict__ buf,
                                                      double *__restrict__ acc, double *__restrict__ last) {
    __shared__ double sh[32];
    pdl_wait();
    const int a = blockIdx.x;
    const double *b = buf + (long long)a * psize;
    double p[4] = {0.0, 0.0, 0.0, 0.0};
    int k = threadIdx.x;
    for (; k + 3 * 1024 < psize; k += 4 * 1024) {
#pragma unroll
        for (int j = 0; j < 4; ++j) p[j] += b[k + 1024 * j];
    }
    for (; k < psize; k += 1024) p[0] += b[k];
    const double s = block_sum<1024>((p[0] + p[1]) + (p[2] + p[3]), sh);
    if (threadIdx.x == 0) {
        acc[a] += s;
        last[a] = s;
    }
}

cudaError_t launch_flux_reduce(int M, int plane_size, const double *buf, double *acc, double *last,
                               cudaStream_t st) {
    return launch_pdl(k_flux_reduce, M, 1024, 0, st, plane_size, buf, acc, last);
}

__global__ void __launch_bounds__(NT) k_reduce_partial(const double *__restrict__ x, long long n, long long chunk,
                                                       double *__restrict__ partial) {
    __shared__ double sh[32];
    const long long b0 = (long long)blockIdx.x * chunk;
    const long long b1 = min(n, b0 + chunk);
    double s = 0.0, mx = 0.0;
    for (long long k = b0 + threadIdx.x; k < b1; k += NT) {
        s += x[k];
        mx = fmax(mx, fabs(x[k]));
    }
    s = block_sum<NT>(s, sh);
    mx = block_max<NT>(mx, sh);
    if (threadIdx.x == 0) {
        partial[2 * blockIdx.x] = s;
        partial[2 * blockIdx.x + 1] = mx;
    }
}

__global__ void __launch_bounds__(1024) k_reduce_final(const double *__restrict__ partial, int np,
                                                       double *__restrict__ out) {
    __shared__ double sh[32];
    double s = 0.0, mx = 0.0;
    for (int k = threadIdx.x; k < np; k += 1024) {
        s += partial[2 * k];
        mx = fmax(mx, partial[2 * k + 1]);
    }
    s = block_sum<1024>(s, sh);
    mx = block_max<1024>(mx, sh);
    if (threadIdx.x == 0) {
        out[0] = s;
        out[1] = mx;
    }
}

cudaError_t launch_reduce(const double *x, long long n, double *partial, int npartial, double *out,
                          cudaStream_t st) {
    long long chunk = (n + npartial - 1) / npartial;
    if (chunk < 1) chunk = 1;
    int nb = (int)((n + chunk - 1) / chunk);
    if (nb < 1) nb = 1;
    k_reduce_partial<<<nb, NT, 0, st>>>(x, n, chunk, partial);
    k_reduce_final<<<1, 1024, 0, st>>>(partial, nb, out);
    return cudaGetLastError();
}

template <typename T>
__global__ void k_to_f64(const T *__restrict__ src, long long n, double *__restrict__ dst) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) dst[i] = (double)src[i];
}

cudaError_t launch_to_f64(bool fp64, const void *src, long long n, double *dst, cudaStream_t st) {
    unsigned nb = (unsigned)((n + NT - 1) / NT);
    if (fp64)
        k_to_f64<double><<<nb, NT, 0, st>>>((const double *)src, n, dst);
    else
        k_to_f64<float><<<nb, NT, 0, st>>>((const float *)src, n, dst);
    return cudaGetLastError();
}

template <typename T>
__global__ void k_unpad(Grid g, const T *__restrict__ pad, double *__restrict__ dst) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.N) return;
    int x, y, z;
    node_xyz(g, i, x, y, z);
    dst[i] = (double)pad[pidx(g, x, y, z)];
}

cudaError_t launch_unpad(bool fp64, const Grid &g, const void *pad, double *dst, cudaStream_t st) {
    unsigned nb = (unsigned)((g.N + NT - 1) / NT);
    if (fp64)
        k_unpad<double><<<nb, NT, 0, st>>>(g, (const double *)pad, dst);
    else
        k_unpad<float><<<nb, NT, 0, st>>>(g, (const float *)pad, dst);
    return cudaGetLastError();
}

// Velocity u = sum_sel J / sum_sel n (sel: species s, or all for s < 0), 0 where n = 0.
__global__ void k_velocity(int M, long long N, int s, const double *__restrict__ n, const double *__restrict__ J,
                           double *__restrict__ u, double *__restrict__ speed) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    double nn = 0.0, j0 = 0.0, j1 = 0.0, j2 = 0.0;
    for (int a = 0; a < M; ++a) {
        if (s >= 0 && a != s) continue;
        nn += n[(long long)a * N + i];
        j0 += J[((long long)a * 3 + 0) * N + i];
        j1 += J[((long long)a * 3 + 1) * N + i];
        j2 += J[((long long)a * 3 + 2) * N + i];
    }
    const double r = nn > 0.0 ? 1.0 / nn : 0.0;
    if (u) {
        u[i] = j0 * r;
        u[N + i] = j1 * r;
        u[2 * N + i] = j2 * r;
    }
    if (speed) speed[i] = sqrt(j0 * j0 + j1 * j1 + j2 * j2) * r;
}

cudaError_t launch_velocity(int M, long long N, int s, const double *n, const double *J, double *u, double *speed,
                            cudaStream_t st) {
    k_velocity<<<(unsigned)((N + NT - 1) / NT), NT, 0, st>>>(M, N, s, n, J, u, speed);
    return cudaGetLastError();
}

// Self-test of the failure detector of the TMA kernels: one thread arms an mbarrier for 16 bytes that
// no copy will deliver (none is issued, so nothing is in flight) and waits on it with the kernels'
// bounded wait, limited to `polls` polls.  The wait gives up and records ERR_TMA_WAIT in the error
// word, as a kernel whose copy never completed would; the barrier is invalidated before the CTA exits.
__global__ void k_wait_probe(int *err, long long polls) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
        mbar_arrive_expect_tx(&bar, 16u);
        mbar_wait_bounded(&bar, 0u, err, polls);
        mbar_inval(&bar);
    }
}

cudaError_t launch_wait_probe(int *err, long long polls, cudaStream_t st) {
    k_wait_probe<<<1, 32, 0, st>>>(err, polls);
    return cudaGetLastError();
}

}  // namespace lbe
