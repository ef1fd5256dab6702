// kernels.cuh -- device code of the lattice Boltzmann solver (sm_103a).
//
// Hot path: one fused pull-stream + BGK-collide kernel per time step (Sec. 6, eq. "LBE update
// scheme").  Populations live in structure-of-arrays layout, one array per velocity, x fastest,
// in a ping-pong pair of buffers.  With SoA and a pull step every stored population that a step
// changes (all but the rest ones for most sets, see rest_static) is read exactly once and written exactly
// once, so DRAM traffic equals the algorithmic 2 * sizeof(storage) bytes per such population
// without any shared-memory staging:
//   - each thread owns V consecutive cells of one x-row (one 16-byte vector per velocity);
//   - a velocity with c_x = 0 is a plain aligned vector load from row (y - c_y, z - c_z);
//   - c_x = +1 / -1 shifts the vector by one element: the missing element comes from the
//     neighbouring lane by warp shuffle, or by a scalar load at a row start or warp edge.
// The collision works on per-shell sums (all weights, additional energies and coefficients of
// the velocity sets depend on |c_i|^2 only), with the whole moment -> equilibrium -> relaxation
// chain folded on the host into two small matrices (see CollideCoef).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include <type_traits>
#include <utility>

#include "velsets.cuh"

namespace lee {

constexpr unsigned kFull = 0xffffffffu;

// ---------------------------------------------------------------------------------------------
// compile-time loops
// ---------------------------------------------------------------------------------------------
template <class F, int... Is>
__device__ __forceinline__ void static_for_impl(F &&f, std::integer_sequence<int, Is...>) {
    (f(std::integral_constant<int, Is>{}), ...);
}
template <int N, class F>
__device__ __forceinline__ void static_for(F &&f) {
    static_for_impl(f, std::make_integer_sequence<int, N>{});
}

template <class S>
__host__ __device__ constexpr bool shell_present(int s) {
    for (int i = 0; i < S::Q; ++i)
        if (S::shell(i) == s) return true;
    return false;
}

// ---------------------------------------------------------------------------------------------
// storage types
// ---------------------------------------------------------------------------------------------
template <class T>
struct Store;
template <>
struct Store<double> {
    using C = double;  // collision arithmetic type
    static constexpr bool scaled = false;
    __device__ static double load(double v) { return v; }
    __device__ static double make(double v) { return v; }
};
template <>
struct Store<float> {
    using C = float;
    static constexpr bool scaled = false;
    __device__ static float load(float v) { return v; }
    __device__ static float make(float v) { return v; }
};
template <>
struct Store<__half> {
    using C = float;
    static constexpr bool scaled = true;  // stores S * g / f*
    __device__ static float load(__half v) { return __half2float(v); }
    __device__ static __half make(float v) { return __float2half_rn(v); }
};
template <>
struct Store<__nv_bfloat16> {
    using C = float;
    static constexpr bool scaled = true;
    __device__ static float load(__nv_bfloat16 v) { return __bfloat162float(v); }
    __device__ static __nv_bfloat16 make(float v) { return __float2bfloat16_rn(v); }
};

template <int BYTES>
struct Raw;
template <>
struct Raw<16> { using type = uint4; };
template <>
struct Raw<8> { using type = uint2; };
template <>
struct Raw<4> { using type = unsigned int; };
template <>
struct Raw<2> { using type = unsigned short; };

// V consecutive elements starting at p (p aligned to V * sizeof(T)), read-only path.
template <class T, int V>
__device__ __forceinline__ void load_vec(const T *__restrict__ p, typename Store<T>::C (&out)[V]) {
    if constexpr (V * sizeof(T) == 8 && sizeof(T) == 8) {
        out[0] = Store<T>::load(__ldg(p));
    } else {
        using R = typename Raw<V * sizeof(T)>::type;
        union {
            R r;
            T e[V];
        } u;
        u.r = __ldg(reinterpret_cast<const R *>(p));
#pragma unroll
        for (int k = 0; k < V; ++k) out[k] = Store<T>::load(u.e[k]);
    }
}

template <class T, int V>
__device__ __forceinline__ void store_vec(T *__restrict__ p, const typename Store<T>::C (&in)[V]) {
    if constexpr (V * sizeof(T) == 8 && sizeof(T) == 8) {
        *p = Store<T>::make(in[0]);
    } else {
        using R = typename Raw<V * sizeof(T)>::type;
        union {
            R r;
            T e[V];
        } u;
#pragma unroll
        for (int k = 0; k < V; ++k) u.e[k] = Store<T>::make(in[k]);
        *reinterpret_cast<R *>(p) = u.r;
    }
}

// ---------------------------------------------------------------------------------------------
// kernel parameters
// ---------------------------------------------------------------------------------------------
struct GridDesc {
    int nx, ny, nz;
    int nxc;            // chunks per row = nx / V
    long long nchunks;  // nxc * ny * nz
    long long pitch;    // elements between consecutive velocity arrays
};

// (xc, y, z) of chunk c = xc + nxc (y + ny z): two 32-bit unsigned divisions while the grid has
// fewer than 2^32 chunks (a warp-uniform test), 64-bit divisions beyond.
__device__ __forceinline__ void chunk_coords(long long c, const GridDesc &gd, int &xc, int &y, int &z) {
    if (gd.nchunks <= 0xFFFFFFFFLL) {
        const unsigned u = (unsigned)c, nxc = (unsigned)gd.nxc, ny = (unsigned)gd.ny;
        const unsigned row = u / nxc;
        xc = (int)(u - row * nxc);
        const unsigned zz = row / ny;
        y = (int)(row - zz * ny);
        z = (int)zz;
    } else {
        const long long row = c / gd.nxc;
        xc = (int)(c - row * gd.nxc);
        const long long zz = row / gd.ny;
        y = (int)(row - zz * gd.ny);
        z = (int)zz;
    }
}

// Collision folded into shell space.  With P_s = sum_{i in shell s} g_i and
// J_s = sum_{i in shell s} c_i g_i, the post-collision population of velocity i in shell t is
//     g*_i = (1 - w) g_i + sum_s M[t][s] P_s + c_i . (sum_s N[t][s] J_s),     w = 1/tau,
// where M and N contain w, f*, the coefficients a1, a2, b, c1, c2, gamma, theta0, rho0 and the
// energies (|c|^2 + beta)/2 (built by the host; exact algebra of Secs. 4-6).
// Conservation of rho', j and the energy moment is an exact identity between these coefficients.
// To keep it exact in FP32 arithmetic, every coefficient is derived from the already rounded w,
// 1 - w is formed in the arithmetic type (exact for 1/2 <= w <= 2), and M is carried as a pair
// M + Mlo (Mlo = the rounding residual of M, zero when M is representable); N is w times a
// power of two for every set and needs no residual.  Rounding of the coefficients then adds no
// systematic drift; only the (unbiased) rounding of the arithmetic remains.
template <class C>
struct CollideCoef {
    C one_minus_omega;
    C M[4][4];
    C Mlo[4][4];
    C N[4][4];
};

// What a step does at the edges of its grid: wraps around, lets zeros enter, damps a frame of cells too (sponge_w of
// them), or lets the populations `ghost` enter (2D).  Every kind has its own instances of the step kernels: the launches of
// open grids are short, and in one instance for all of them each paid for the others' code (D2Q5 FP32, us per step,
// zero edge / frame: 137x197 2.21 / 2.62 in one instance, 1.42 / 1.59 so; 1024^2 4.87 / 6.20 and 3.93 / 4.30).
enum Edge { kWrapEdge, kZeroEdge, kFrameEdge, kGhostEdge };
template <class C>
struct OpenEdge {
    int sponge_w;
    C sponge_smax;
    const C *ghost;      // [4][L] entering populations, or nullptr = zeros
    int ghost_L;
    int skip_border;     // leave the border cells unwritten (the learned edge's kernels own them)
};
template <class C>
__device__ __forceinline__ bool in_frame(int x, int cells, int y, int z, const GridDesc &gd, int D, const OpenEdge<C> &ob) {
    const int w = ob.sponge_w;
    return x < w || x + cells > gd.nx - w || (D >= 2 && (y < w || y >= gd.ny - w)) || (D >= 3 && (z < w || z >= gd.nz - w));
}

// ---------------------------------------------------------------------------------------------
// collision of one cell (index K of the per-thread vector)
// ---------------------------------------------------------------------------------------------
template <class S>
__host__ __device__ constexpr int first_in_shell(int s) {
    for (int i = 0; i < S::Q; ++i)
        if (S::shell(i) == s) return i;
    return -1;
}
template <class S>
__host__ __device__ constexpr int first_on_axis(int s, int a) {
    for (int i = 0; i < S::Q; ++i)
        if (S::shell(i) == s && S::c(i, a) != 0) return i;
    return -1;
}
template <class S>
__host__ __device__ constexpr int first_present_shell(int from) {
    for (int s = from; s < 4; ++s)
        if (shell_present<S>(s)) return s;
    return -1;
}

template <class S>
__host__ __device__ constexpr int moving_shells() {
    int n = 0;
    for (int s = 1; s < 4; ++s) n += shell_present<S>(s) ? 1 : 0;
    return n;
}

// Sets whose moving velocities share one shell (all but D3Q19).  Mass is P_0 + P_1 and energy is
// proportional to P_1, so the collision conserves the shell sums P_0 and P_1 one by one:
// mhat[0] = (1, 0) and mhat[1] = (0, 1/q_1) in the folded coefficients.  Two things follow.
//  - The rest population of a cell never changes (only a sponge frame damps it), so a step neither
//    reads nor writes it: both state copies hold it, written when the state is set.  A D2Q5 FP32 step
//    moves 32 bytes per cell instead of 40, a D3Q7 one 48 instead of 56.
//  - The moving populations collide among themselves.
template <class S>
__host__ __device__ constexpr bool rest_static() {
    return moving_shells<S>() == 1;
}
// Whether a step changes velocity i (velocity 0 is the rest one in every set).
template <class S>
__host__ __device__ constexpr bool carried(int i) {
    return !(rest_static<S>() && S::shell(i) == 0);
}
// Whether shell s takes part in the collision's sums.
template <class S>
__host__ __device__ constexpr bool mixes(int s) {
    return shell_present<S>(s) && !(rest_static<S>() && s == 0);
}
template <class S, class F>
__device__ __forceinline__ void static_for_carried(F &&f) {
    static_for<S::Q>([&](auto I) {
        if constexpr (carried<S>(decltype(I)::value)) f(I);
    });
}

// Rest and axis velocities only (D1Q3, D2Q5, D3Q7 and the diatomic sets).  There the momentum part of
// the equilibrium, f*_1 (b / rho0) c_i . J = (g_+a - g_-a) / 2, is the odd part of the pair itself for
// every set of Sec. 8, so relaxation leaves the odd parts alone and
//     g*_+-a = g_+-a + (w / 2D) (P_1 - D s_a),     s_a = g_+a + g_-a,
// which is 7 operations per cell for D2Q5 (22 in the matrix form) and 14 for D3Q7, and nothing at all
// for D1Q3 (H = I, Sec. 8.1).  Its roundings are fewer than the matrix form's (FP64, D3Q7 diatomic, 50
// steps against 80-bit arithmetic: 7e-17 instead of 6e-15); the corrections of a cell add up to zero
// whatever w / 2D rounds to, so that coefficient needs no residual.  FP64 steps are bound by GB300's
// FP64 pipe, so there it pays most: D2Q5 FP64 2048^2 28.1 -> 71 GLUPS, D3Q7 diatomic FP64 193x161x135
// 20.5 -> 36 GLUPS.
template <class S>
__host__ __device__ constexpr bool axis_set() {
    bool axis = rest_static<S>() && shell_present<S>(1) && S::Q == 2 * S::D + 1;
    for (int a = 0; a < S::D; ++a) axis = axis && S::c(1 + 2 * a, a) == 1 && S::c(2 + 2 * a, a) == -1;
    return axis;
}

// Every rounding is spelled out so that no result depends on the compiler's contraction of a
// multiply and an add: with one moving shell the momentum term of velocity i is one fused
// multiply-add per axis, eq = fma(+-N[t][s1], J[s1][a], eq); with several moving shells the sums
// KJ[t][a] = sum_s N[t][s] J[s][a] (a chain of fused multiply-adds) are added to eq.
template <class S, int K, class C, int V>
__device__ __forceinline__ void collide_shells_cell(const C (&g)[S::Q][V], C (&out)[S::Q][V], const CollideCoef<C> &cf) {
    // Accumulators start at -0.0 so that the first addition folds away exactly.
    C P[4] = {C(-0.0), C(-0.0), C(-0.0), C(-0.0)};
    C J[4][3];
#pragma unroll
    for (int s = 0; s < 4; ++s) J[s][0] = J[s][1] = J[s][2] = C(-0.0);
    static_for_carried<S>([&](auto I) {
        constexpr int i = decltype(I)::value;
        constexpr int s = S::shell(i);
        const C v = g[i][K];
        P[s] += v;
        static_for<3>([&](auto A) {
            constexpr int a = decltype(A)::value;
            if constexpr (S::c(i, a) == 1) J[s][a] += v;
            if constexpr (S::c(i, a) == -1) J[s][a] -= v;
        });
    });
    C B[4], KJ[4][3];
    static_for<4>([&](auto T) {
        constexpr int t = decltype(T)::value;
        if constexpr (mixes<S>(t)) {
            C acc = C(-0.0);
            if constexpr (std::is_same<C, float>::value) {
                static_for<4>([&](auto Sx) {
                    constexpr int s = decltype(Sx)::value;
                    if constexpr (mixes<S>(s)) acc = fma(cf.Mlo[t][s], P[s], acc);
                });
            }
            static_for<4>([&](auto Sx) {
                constexpr int s = decltype(Sx)::value;
                if constexpr (mixes<S>(s)) acc = fma(cf.M[t][s], P[s], acc);
            });
            B[t] = acc;
            if constexpr (t > 0 && moving_shells<S>() > 1) {
                static_for<S::D>([&](auto A) {
                    constexpr int a = decltype(A)::value;
                    C kj = C(-0.0);
                    static_for<4>([&](auto Sx) {
                        constexpr int s = decltype(Sx)::value;
                        if constexpr (s > 0 && shell_present<S>(s)) kj = fma(cf.N[t][s], J[s][a], kj);
                    });
                    KJ[t][a] = kj;
                });
            }
        }
    });
    static_for_carried<S>([&](auto I) {
        constexpr int i = decltype(I)::value;
        constexpr int t = S::shell(i);
        C eq = B[t];
        static_for<S::D>([&](auto A) {
            constexpr int a = decltype(A)::value;
            constexpr int c = S::c(i, a);
            if constexpr (c != 0 && moving_shells<S>() == 1) {
                constexpr int s1 = first_present_shell<S>(1);
                eq = fma(c == 1 ? cf.N[t][s1] : -cf.N[t][s1], J[s1][a], eq);
            } else if constexpr (c == 1) {
                eq += KJ[t][a];
            } else if constexpr (c == -1) {
                eq -= KJ[t][a];
            }
        });
        out[i][K] = fma(cf.one_minus_omega, g[i][K], eq);
    });
}

template <class S, int K, class C, int V>
__device__ __forceinline__ void collide_axis_cell(const C (&g)[S::Q][V], C (&out)[S::Q][V], const CollideCoef<C> &cf) {
    const C w = cf.M[1][1];  // w / 2D
    if constexpr (S::D == 1) {
        out[1][K] = g[1][K];
        out[2][K] = g[2][K];
    } else if constexpr (S::D == 2) {
        const C d = (g[3][K] + g[4][K]) - (g[1][K] + g[2][K]);
        out[1][K] = fma(w, d, g[1][K]);
        out[2][K] = fma(w, d, g[2][K]);
        out[3][K] = fma(-w, d, g[3][K]);
        out[4][K] = fma(-w, d, g[4][K]);
    } else {
        const C sx = g[1][K] + g[2][K], sy = g[3][K] + g[4][K], sz = g[5][K] + g[6][K];
        const C P = (sx + sy) + sz;
        const C tx = fma(C(-3), sx, P), ty = fma(C(-3), sy, P), tz = fma(C(-3), sz, P);
        out[1][K] = fma(w, tx, g[1][K]);
        out[2][K] = fma(w, tx, g[2][K]);
        out[3][K] = fma(w, ty, g[3][K]);
        out[4][K] = fma(w, ty, g[4][K]);
        out[5][K] = fma(w, tz, g[5][K]);
        out[6][K] = fma(w, tz, g[6][K]);
    }
}

template <class S, int K, class C, int V>
__device__ __forceinline__ void collide_cell(const C (&g)[S::Q][V], C (&out)[S::Q][V], const CollideCoef<C> &cf) {
    if constexpr (rest_static<S>()) out[0][K] = g[0][K];
    if constexpr (axis_set<S>()) collide_axis_cell<S, K>(g, out, cf);
    else collide_shells_cell<S, K>(g, out, cf);
}

// FP32 collision of two cells (K, K+1) at once with the packed f32x2 add, mul and fma of sm_100
// and later.  Every packed operation rounds each half exactly like the scalar operation it
// replaces in collide_cell (a - b is a + (-b); a first accumulation into -0.0 is the value itself,
// or a plain product for the fma chains), so the result is the same bit for bit with half the FP
// instructions.
__device__ __forceinline__ float2 splat2(float c) { return make_float2(c, c); }
__device__ __forceinline__ float2 neg2(float2 v) { return make_float2(-v.x, -v.y); }

template <class S, int K, int V>
__device__ __forceinline__ void collide_shells_pair(const float (&g)[S::Q][V], float (&out)[S::Q][V],
                                             const CollideCoef<float> &cf) {
    float2 P[4], J[4][3];
    static_for_carried<S>([&](auto I) {
        constexpr int i = decltype(I)::value;
        constexpr int s = S::shell(i);
        const float2 v = make_float2(g[i][K], g[i][K + 1]);
        if constexpr (i == first_in_shell<S>(s)) P[s] = v;
        else P[s] = __fadd2_rn(P[s], v);
        static_for<3>([&](auto A) {
            constexpr int a = decltype(A)::value;
            constexpr int c = S::c(i, a);
            if constexpr (c != 0) {
                const float2 sv = c == 1 ? v : neg2(v);
                if constexpr (i == first_on_axis<S>(s, a)) J[s][a] = sv;
                else J[s][a] = __fadd2_rn(J[s][a], sv);
            }
        });
    });
    float2 B[4], KJ[4][3];
    static_for<4>([&](auto T) {
        constexpr int t = decltype(T)::value;
        if constexpr (mixes<S>(t)) {
            constexpr int s0 = first_present_shell<S>(rest_static<S>() ? 1 : 0);
            float2 acc;
            static_for<4>([&](auto Sx) {
                constexpr int s = decltype(Sx)::value;
                if constexpr (mixes<S>(s)) {
                    if constexpr (s == s0) acc = __fmul2_rn(splat2(cf.Mlo[t][s]), P[s]);
                    else acc = __ffma2_rn(splat2(cf.Mlo[t][s]), P[s], acc);
                }
            });
            static_for<4>([&](auto Sx) {
                constexpr int s = decltype(Sx)::value;
                if constexpr (mixes<S>(s)) acc = __ffma2_rn(splat2(cf.M[t][s]), P[s], acc);
            });
            B[t] = acc;
            if constexpr (t > 0 && moving_shells<S>() > 1) {
                constexpr int s1 = first_present_shell<S>(1);
                static_for<S::D>([&](auto A) {
                    constexpr int a = decltype(A)::value;
                    float2 kj;
                    static_for<4>([&](auto Sx) {
                        constexpr int s = decltype(Sx)::value;
                        if constexpr (s > 0 && shell_present<S>(s)) {
                            if constexpr (s == s1) kj = __fmul2_rn(splat2(cf.N[t][s]), J[s][a]);
                            else kj = __ffma2_rn(splat2(cf.N[t][s]), J[s][a], kj);
                        }
                    });
                    KJ[t][a] = kj;
                });
            }
        }
    });
    const float2 omm = splat2(cf.one_minus_omega);
    static_for_carried<S>([&](auto I) {
        constexpr int i = decltype(I)::value;
        constexpr int t = S::shell(i);
        float2 eq = B[t];
        static_for<S::D>([&](auto A) {
            constexpr int a = decltype(A)::value;
            constexpr int c = S::c(i, a);
            if constexpr (c != 0 && moving_shells<S>() == 1) {
                constexpr int s1 = first_present_shell<S>(1);
                eq = __ffma2_rn(splat2(c == 1 ? cf.N[t][s1] : -cf.N[t][s1]), J[s1][a], eq);
            } else if constexpr (c == 1) {
                eq = __fadd2_rn(eq, KJ[t][a]);
            } else if constexpr (c == -1) {
                eq = __fadd2_rn(eq, neg2(KJ[t][a]));
            }
        });
        const float2 r = __ffma2_rn(omm, make_float2(g[i][K], g[i][K + 1]), eq);
        out[i][K] = r.x;
        out[i][K + 1] = r.y;
    });
}

template <class S, int K, int V>
__device__ __forceinline__ void collide_axis_pair(const float (&g)[S::Q][V], float (&out)[S::Q][V],
                                                  const CollideCoef<float> &cf) {
    const float w = cf.M[1][1];
    auto in = [&](int i) { return make_float2(g[i][K], g[i][K + 1]); };
    auto put = [&](int i, float c, float2 t) {
        const float2 r = __ffma2_rn(splat2(c), t, in(i));
        out[i][K] = r.x;
        out[i][K + 1] = r.y;
    };
    if constexpr (S::D == 1) {
#pragma unroll
        for (int i = 1; i < 3; ++i) {
            out[i][K] = g[i][K];
            out[i][K + 1] = g[i][K + 1];
        }
    } else if constexpr (S::D == 2) {
        const float2 d = __fadd2_rn(__fadd2_rn(in(3), in(4)), neg2(__fadd2_rn(in(1), in(2))));
        put(1, w, d);
        put(2, w, d);
        put(3, -w, d);
        put(4, -w, d);
    } else {
        const float2 sx = __fadd2_rn(in(1), in(2)), sy = __fadd2_rn(in(3), in(4)), sz = __fadd2_rn(in(5), in(6));
        const float2 P = __fadd2_rn(__fadd2_rn(sx, sy), sz), m3 = splat2(-3.0f);
        const float2 tx = __ffma2_rn(m3, sx, P), ty = __ffma2_rn(m3, sy, P), tz = __ffma2_rn(m3, sz, P);
        put(1, w, tx);
        put(2, w, tx);
        put(3, w, ty);
        put(4, w, ty);
        put(5, w, tz);
        put(6, w, tz);
    }
}

template <class S, int K, int V>
__device__ __forceinline__ void collide_pair(const float (&g)[S::Q][V], float (&out)[S::Q][V],
                                             const CollideCoef<float> &cf) {
    static_assert(K + 1 < V, "a pair needs two cells");
    if constexpr (rest_static<S>()) {
        out[0][K] = g[0][K];
        out[0][K + 1] = g[0][K + 1];
    }
    if constexpr (axis_set<S>()) collide_axis_pair<S, K>(g, out, cf);
    else collide_shells_pair<S, K>(g, out, cf);
}

// All V cells of a chunk: FP32 pairs on the packed path, anything else one cell at a time (both
// give the same bits).
template <class S, bool PACK = true, class C, int V>
__device__ __forceinline__ void collide_chunk(const C (&g)[S::Q][V], C (&out)[S::Q][V], const CollideCoef<C> &cf) {
    if constexpr (PACK && std::is_same<C, float>::value && V % 2 == 0) {
        static_for<V / 2>([&](auto Kx) { collide_pair<S, 2 * decltype(Kx)::value>(g, out, cf); });
    } else {
        static_for<V>([&](auto Kx) { collide_cell<S, decltype(Kx)::value>(g, out, cf); });
    }
}

template <class C>
__device__ __forceinline__ C sponge_factor(int x, int y, int z, const GridDesc &gd, int D, int w, C smax) {
    int d = 0;
    const int p[3] = {x, y, z};
    const int n[3] = {gd.nx, gd.ny, gd.nz};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (a < D) {
            d = max(d, w - p[a]);
            d = max(d, p[a] - (n[a] - 1 - w));
        }
    }
    if (d <= 0) return C(1);
    const C r = C(d) / C(w);
    return fma(-(smax * r), r, C(1));  // 1 - smax r^2, one rounding of the product (smax r) r
}

// ---------------------------------------------------------------------------------------------
// fused pull-stream + collide, one time step
// ---------------------------------------------------------------------------------------------
// One thread's share of a step: V cells starting at chunk `raw` of the grid gd.  All 32 lanes of
// the warp must call this together (warp shuffles); lanes with raw >= nchunks compute on a clamped
// chunk and store nothing.  CUT (a slab of a larger periodic domain, cut along its last axis: y in
// 2D, z in 3D): along that axis nothing wraps -- the rows just before and after the grid are read
// where they lie in memory, in the halo planes the caller keeps there -- and every other axis is
// periodic.
template <class S, class T, int V, Edge EDGE, bool CUT = false>
__device__ __forceinline__ void stream_collide_chunk(const T *__restrict__ src, T *__restrict__ dst, const GridDesc &gd,
                                                     const CollideCoef<typename Store<T>::C> &cf,
                                                     const OpenEdge<typename Store<T>::C> &ob, long long raw) {
    constexpr bool OPEN = EDGE != kWrapEdge;
    static_assert(!(CUT && OPEN), "a slab is periodic across its cut faces' neighbours");
    static_assert(EDGE != kGhostEdge || S::D == 2, "entering populations of a 2D grid");
    using C = typename Store<T>::C;
    const bool active = raw < gd.nchunks;
    const long long chunk = active ? raw : gd.nchunks - 1;
    const int lane = threadIdx.x & 31;
    int xc, y, z;
    chunk_coords(chunk, gd, xc, y, z);
    const int x0 = xc * V;
    const bool has_left = (lane > 0) && (xc > 0);
    const bool has_right = (lane < 31) && (xc < gd.nxc - 1);

    // The frame damps rest populations that a step leaves alone elsewhere.  In 2D those of the chunks that touch it are
    // read, after the pulls (32x32 FP16 2.32 us per step; before them 2.75); in 3D, where a frame is most of a small
    // grid, those of all, before the pulls (D3Q13 100^3 FP32 16.3; of the frame's chunks 17.2; after the pulls 17.4).
    constexpr bool REST = EDGE == kFrameEdge && rest_static<S>();
    [[maybe_unused]] C rest[V];
    [[maybe_unused]] const bool framed = !REST || S::D == 3 || in_frame(x0, V, y, z, gd, S::D, ob);
    auto load_rest = [&] { load_vec<T, V>(src + ((long long)z * gd.ny + y) * gd.nx + x0, rest); };
    if constexpr (REST && S::D == 3) load_rest();
    C pull[S::Q][V];
    static_for_carried<S>([&](auto I) {
        constexpr int i = decltype(I)::value;
        constexpr int cx = S::c(i, 0), cy = S::c(i, 1), cz = S::c(i, 2);
        int ys = y - cy, zs = z - cz;
        bool row_out = false;
        if constexpr (cy != 0 && !(CUT && S::D == 2)) {
            if (ys < 0) { if constexpr (OPEN) row_out = true; else ys += gd.ny; }
            if (ys >= gd.ny) { if constexpr (OPEN) row_out = true; else ys -= gd.ny; }
        }
        if constexpr (cz != 0 && !(CUT && S::D == 3)) {
            if (zs < 0) { if constexpr (OPEN) row_out = true; else zs += gd.nz; }
            if (zs >= gd.nz) { if constexpr (OPEN) row_out = true; else zs -= gd.nz; }
        }
        // (rows outside the grid: the cell's own is read for them, so that no load waits on a branch)
        if constexpr (OPEN && cy != 0) ys = row_out ? y : ys;
        if constexpr (OPEN && cz != 0) zs = row_out ? z : zs;
        const T *rowp = src + (long long)i * gd.pitch + ((long long)zs * gd.ny + ys) * gd.nx;
        C v[V];
        load_vec<T, V>(rowp + x0, v);
        if (OPEN && (cy != 0 || cz != 0) && row_out) {
#pragma unroll
            for (int k = 0; k < V; ++k) v[k] = C(0);
            if constexpr (EDGE == kGhostEdge && cx == 0) {
                if (ob.ghost != nullptr) {  // entering through the bottom (c_y = +1) or top edge
                    const C *gp = ob.ghost + (cy == 1 ? 2 : 3) * ob.ghost_L + x0;
#pragma unroll
                    for (int k = 0; k < V; ++k) v[k] = gp[k];
                }
            }
        }
        if constexpr (cx == 0) {
#pragma unroll
            for (int k = 0; k < V; ++k) pull[i][k] = v[k];
        } else if constexpr (cx == 1) {
            const C prev = __shfl_up_sync(kFull, v[V - 1], 1);
            C left;
            if (has_left) {
                left = prev;
            } else {
                int xs = x0 - 1;
                const bool out = xs < 0;
                if (out) xs = OPEN ? x0 : xs + gd.nx;
                left = Store<T>::load(rowp[xs]);
                if (OPEN && (out || row_out)) left = C(0);
                if constexpr (EDGE == kGhostEdge && cy == 0) {
                    if (out && ob.ghost != nullptr) left = ob.ghost[0 * ob.ghost_L + y];
                }
            }
            pull[i][0] = left;
#pragma unroll
            for (int k = 1; k < V; ++k) pull[i][k] = v[k - 1];
        } else {
            const C next = __shfl_down_sync(kFull, v[0], 1);
            C right;
            if (has_right) {
                right = next;
            } else {
                int xs = x0 + V;
                const bool out = xs >= gd.nx;
                if (out) xs = OPEN ? x0 : xs - gd.nx;
                right = Store<T>::load(rowp[xs]);
                if (OPEN && (out || row_out)) right = C(0);
                if constexpr (EDGE == kGhostEdge && cy == 0) {
                    if (out && ob.ghost != nullptr) right = ob.ghost[1 * ob.ghost_L + y];
                }
            }
#pragma unroll
            for (int k = 0; k < V - 1; ++k) pull[i][k] = v[k + 1];
            pull[i][V - 1] = right;
        }
    });

    if constexpr (REST && S::D < 3) {
        if (framed) load_rest();
    }
    C post[S::Q][V];
    // one cell at a time: this kernel streams at the memory bound, and the packed f32x2 pairs
    // (same bits) cost it 9 to 12 registers and occupancy
    collide_chunk<S, false>(pull, post, cf);

    if constexpr (EDGE == kFrameEdge) {
        if (REST ? framed : ob.sponge_w > 0) {
#pragma unroll
            for (int k = 0; k < V; ++k) {
                const C damp = sponge_factor<C>(x0 + k, y, z, gd, S::D, ob.sponge_w, ob.sponge_smax);
                if constexpr (REST) rest[k] *= damp;
#pragma unroll
                for (int i = REST ? 1 : 0; i < S::Q; ++i) post[i][k] *= damp;
            }
            if (REST && active) store_vec<T, V>(dst + ((long long)z * gd.ny + y) * gd.nx + x0, rest);
        }
    }

    if (active) {
        T *outp = dst + ((long long)z * gd.ny + y) * gd.nx + x0;
        if constexpr (EDGE == kGhostEdge) {
            if (ob.skip_border) {
                if (y == 0 || y == gd.ny - 1) return;
                if (x0 == 0 || x0 + V >= gd.nx) {  // a chunk that holds x = 0 or x = nx - 1
                    static_for_carried<S>([&](auto I) {
                        constexpr int i = decltype(I)::value;
#pragma unroll
                        for (int k = 0; k < V; ++k) {
                            if (x0 + k >= 1 && x0 + k <= gd.nx - 2)
                                outp[(long long)i * gd.pitch + k] = Store<T>::make(post[i][k]);
                        }
                    });
                    return;
                }
            }
        }
        static_for_carried<S>([&](auto I) {
            constexpr int i = decltype(I)::value;
            store_vec<T, V>(outp + (long long)i * gd.pitch, post[i]);
        });
    }
}

// All n steps of a small 1D grid in one launch: one block keeps both population copies in
// shared memory (in the storage type, so every step rounds exactly like the global-memory path)
// and synchronises between steps.  Same per-cell arithmetic as k_stream_collide, so the result
// equals n launches of it bit for bit.  The final state is written back to g (in place).
template <class S, class T>
__global__ void __launch_bounds__(1024) k_onchip_1d(T *__restrict__ g, int nx, long long pitch,
                                                    CollideCoef<typename Store<T>::C> cf,
                                                    OpenEdge<typename Store<T>::C> ob, bool open, long long nsteps) {
    using C = typename Store<T>::C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *bufA = reinterpret_cast<T *>(smem_raw);
    T *bufB = bufA + (size_t)S::Q * nx;
    for (int k = threadIdx.x; k < S::Q * nx; k += blockDim.x) bufA[k] = g[(long long)(k / nx) * pitch + k % nx];
    __syncthreads();
    const GridDesc gd{nx, 1, 1, nx, nx, nx};
    for (long long step = 0; step < nsteps; ++step) {
        const T *src = (step & 1) ? bufB : bufA;
        T *dst = (step & 1) ? bufA : bufB;
        for (int x = threadIdx.x; x < nx; x += blockDim.x) {
            C pull[S::Q][1], post[S::Q][1];
            static_for<S::Q>([&](auto I) {
                constexpr int i = decltype(I)::value;
                int xs = x - S::c(i, 0);
                bool out = false;
                if (xs < 0) { if (open) out = true; else xs += nx; }
                if (xs >= nx) { if (open) out = true; else xs -= nx; }
                pull[i][0] = out ? C(0) : Store<T>::load(src[i * nx + xs]);
            });
            collide_cell<S, 0>(pull, post, cf);
            if (open && ob.sponge_w > 0) {
                const C damp = sponge_factor<C>(x, 0, 0, gd, 1, ob.sponge_w, ob.sponge_smax);
#pragma unroll
                for (int i = 0; i < S::Q; ++i) post[i][0] *= damp;
            }
#pragma unroll
            for (int i = 0; i < S::Q; ++i) dst[i * nx + x] = Store<T>::make(post[i][0]);
        }
        __syncthreads();
    }
    const T *fin = (nsteps & 1) ? bufB : bufA;
    for (int k = threadIdx.x; k < S::Q * nx; k += blockDim.x) g[(long long)(k / nx) * pitch + k % nx] = fin[k];
}

// Blocks per SM for which the compiler lays out the kernels of many registers; 0 is its own choice, which is right
// elsewhere (a bound of one block makes it take many more).  us per step, its choice and the bound: D3Q13 FP16
// 160^3 36.7 and 30.7, frame 97 and 52; D3Q13 FP32 160^3 zero edge 71 and 63; frames of D3Q7 FP16 160^3 28 and 23, of
// D3Q9 FP32 160^3 57 and 52.
template <class S, class T, int V, Edge EDGE>
__host__ __device__ constexpr int step_min_blocks() {
    int pulls = 0;  // registers of a thread's pulls
    for (int i = 0; i < S::Q; ++i) pulls += carried<S>(i) ? V * (int)sizeof(typename Store<T>::C) / 4 : 0;
    if (!rest_static<S>() || sizeof(T) == 8) return 0;
    if (pulls > 64) return 2;
    if (EDGE == kWrapEdge) return 0;
    if (V == 8) return pulls > 32 ? 3 : 0;
    return pulls > 32 ? (EDGE == kZeroEdge ? 4 : 0) : pulls == 32 && V == 4 && EDGE == kFrameEdge ? 4 : 0;
}

// One fused time step on one grid: one thread per V-cell chunk.
template <class S, class T, int V, Edge EDGE, bool CUT = false>
__global__ void __launch_bounds__(256, step_min_blocks<S, T, V, EDGE>())
    k_stream_collide(const T *__restrict__ src, T *__restrict__ dst, GridDesc gd, CollideCoef<typename Store<T>::C> cf,
                     OpenEdge<typename Store<T>::C> ob) {
    stream_collide_chunk<S, T, V, EDGE, CUT>(src, dst, gd, cf, ob, (long long)blockIdx.x * blockDim.x + threadIdx.x);
}

__device__ __forceinline__ void prefetch_l2(const void *p) { asm volatile("prefetch.global.L2 [%0];\n" ::"l"(p)); }

// Many independent periodic grids (one per domain) advanced by one launch.  Domain d owns the
// blocks [first_block[d], first_block[d+1]); its populations start at element offset[d] of the
// shared buffers, and it has its own extents and relaxation coefficients (its own tau).  The
// block -> domain map is a table, so a block never straddles two domains.
template <class C>
struct BatchDomain {
    GridDesc gd;
    CollideCoef<C> cf;
    long long offset;
    int first_block;
};

template <class S, class T, int V>
__global__ void __launch_bounds__(512) k_stream_collide_batched(const T *__restrict__ src, T *__restrict__ dst,
                                                                const BatchDomain<typename Store<T>::C> *__restrict__ doms,
                                                                const unsigned short *__restrict__ block_domain) {
    using C = typename Store<T>::C;
    const int d = block_domain[blockIdx.x];
    const BatchDomain<C> &D = doms[d];
    const long long raw = (long long)(blockIdx.x - D.first_block) * blockDim.x + threadIdx.x;
    const OpenEdge<C> none{0, C(0), nullptr, 0};
    stream_collide_chunk<S, T, V, kWrapEdge>(src + D.offset, dst + D.offset, D.gd, D.cf, none, raw);
}

}  // namespace lee
