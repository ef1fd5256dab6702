// aux_kernels.cuh -- auxiliary kernels of the solver (sm_103a): equilibrium initialisation,
// per-cell moments, FP64 reductions, sponge damping of an initial state, FP64 import/export.
// They run once per job, not per time step.
#pragma once

#include "bfp.cuh"

namespace lee {

// ---------------------------------------------------------------------------------------------
// auxiliary kernels: equilibrium initialisation, moments, reductions, FP64 import/export
// ---------------------------------------------------------------------------------------------

// Per-set FP64 constants for the auxiliary kernels (general form of Sec. 5).  The kernels work
// on per-shell sums (every weight and coefficient depends on the shell |c_i|^2 only), so the
// shell factors are folded on the host and each population costs one or two FP64 additions:
//   g_i^eq = eqA[.][s] rho' + eqB[.][s] theta' + eqC[.][s] (c_i . u')   (i in shell s;
//            [0] the population itself, [1] the scaled 16-bit value S g_i / f*_s),
//   with eqA = F (a1 + s c1 / 2), eqB = F (a2 + s c2 / 2), eqC = F b, F = f*_s resp. 1;
//   a stored 16-bit value decodes as g = dec[s] x stored, dec = f*_s / S (enc = 1 / dec);
//   the energy moment weight of shell s is ew[s] = (s + beta_s) / 2;
//   u' = j / rho0 and theta' = kE e - kR rho' with kE = (gamma - 1) / rho0, kR = theta0 / rho0.
// (|c|^2 = s for every velocity of shell s.)
struct SetConsts {
    double rho0, theta0, gamma, a1, a2, b, c1, c2;
    double f[4];     // f* per shell
    double beta[4];  // beta per shell
    double scale;    // 16-bit storage scale S (1 otherwise)
    double eqA[2][4], eqB[2][4], eqC[2][4];
    double dec[4], enc[4], ew[4];
    double te[2][4];  // energy weights of theta': kE ew ([1]: of stored 16-bit values, kE ew dec)
    double inv_rho0, kE, kR;
};

// Shells present in set S, in increasing order, and the compact slot of shell s.
template <class S>
__host__ __device__ constexpr int n_shells() {
    int n = 0;
    for (int s = 0; s < 4; ++s) n += shell_present<S>(s) ? 1 : 0;
    return n;
}
template <class S>
__host__ __device__ constexpr int shell_slot(int s) {
    int n = 0;
    for (int t = 0; t < s; ++t) n += shell_present<S>(t) ? 1 : 0;
    return n;
}

template <class S>
__device__ __forceinline__ double decode(double stored, int i, const SetConsts &k, bool scaled) {
    return scaled ? stored * k.dec[S::shell(i)] : stored;
}

// g_i^eq of one cell for every velocity: per shell two products, per velocity the signed sum of
// the velocity components it moves along and one fused multiply-add.
template <class S, int SC, class F>
__device__ __forceinline__ void equilibrium_cell(double r, double th, const double (&uu)[3], const SetConsts &k, F &&put) {
    double base[4];
    static_for<4>([&](auto Sx) {
        constexpr int s = decltype(Sx)::value;
        if constexpr (shell_present<S>(s)) base[s] = fma(k.eqB[SC][s], th, k.eqA[SC][s] * r);
    });
    static_for<S::Q>([&](auto I) {
        constexpr int i = decltype(I)::value;
        constexpr int s = S::shell(i);
        constexpr bool moving = S::c(i, 0) != 0 || S::c(i, 1) != 0 || S::c(i, 2) != 0;
        if constexpr (!moving) {
            put(i, base[s]);
        } else {
            double cu = 0.0;
            bool first = true;
            static_for<3>([&](auto A) {
                constexpr int a = decltype(A)::value;
                constexpr int c = S::c(i, a);
                if constexpr (c != 0) {
                    const double t = c == 1 ? uu[a] : -uu[a];
                    cu = first ? t : cu + t;
                    first = false;
                }
            });
            put(i, fma(k.eqC[SC][s], cu, base[s]));
        }
    });
}

// The auxiliary kernels are bound by GB300's FP64 pipe (two lanes per clock and SM), which also takes the
// conversions between FP64 and the other types.  They keep FP64's precision with fewer of its
// instructions: conversions and sums run on the integer pipes where that is exact.

// (float)v, rounded to nearest even: on the integer pipe where v is a normal FP32 number.
__device__ __forceinline__ float to_f32(double v) {
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    if (((hi >> 20) & 0x7FFu) - 897u < 254u) {
        // half an FP32 unit less one, plus the kept part's last bit, carries exactly where v rounds up
        const unsigned long long r = (((unsigned long long)hi << 32) | lo) + 0x0FFFFFFFull + ((lo >> 29) & 1u);
        const unsigned kept = (unsigned)((r - (896ull << 52)) >> 29);
        return __uint_as_float((kept & 0x7FFFFFFFu) | (hi & 0x80000000u));
    }
    return (float)v;
}
template <class C>
__device__ __forceinline__ C to_store(double v) {
    if constexpr (std::is_same<C, float>::value) return to_f32(v);
    else return v;
}

// Writers of a state copy g also write the rest populations of the sets that leave them alone
// (rest_static) into the other copy, `other`: a step neither reads nor writes them.

// g_i = g_i^eq(rho', u', theta') (Sec. 7 initial condition), encoded into storage type T.
template <class S, class T>
__global__ void k_init_equilibrium(const double *__restrict__ rho, const double *__restrict__ u,
                                   const double *__restrict__ theta, T *__restrict__ g, T *__restrict__ other,
                                   long long cells, long long pitch, SetConsts k) {
    constexpr int SC = Store<T>::scaled ? 1 : 0;
    for (long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x; x < cells; x += (long long)gridDim.x * blockDim.x) {
        double uu[3] = {0.0, 0.0, 0.0};
#pragma unroll
        for (int a = 0; a < S::D; ++a) uu[a] = u[(long long)a * cells + x];
        equilibrium_cell<S, SC>(rho[x], theta[x], uu, k, [&](int i, double v) {
            const T e = Store<T>::make(to_store<typename Store<T>::C>(v));
            g[(long long)i * pitch + x] = e;
            if (rest_static<S>() && i == 0) other[x] = e;
        });
    }
}

// An estimate of the largest |g_i^eq / f*_i| of the initial fields in FP32, and the largest sum of the magnitudes
// that a value was put together from: the estimate is off by less than kInitError times that (a dozen roundings
// of 2^-24 of them).  The host needs the maximum's place between two powers of two only, so this decides it for
// nearly all fields; k_init_maxabs, bound by the FP64 pipe, is left for those where it does not (and for fields
// outside 1e-30 .. 1e30, where the estimate is infinite or small).  NaN is left out as there.  D2Q5, 8192^2 FP16: init_fields
// 3.07 -> 1.91 ms.
struct InitCoef {
    float A[4], B[4], C[4];  // eqA[1], eqB[1], eqC[1] for a scale of 1
};
constexpr double kInitError = 1.0 / (1 << 20);
template <class S>
__global__ void k_init_estimate(const double *__restrict__ rho, const double *__restrict__ u,
                                const double *__restrict__ theta, long long cells, InitCoef k,
                                unsigned int *__restrict__ maxbits) {
    float most = 0.f, sum = 0.f;
    for (long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x; x < cells; x += (long long)gridDim.x * blockDim.x) {
        const float r = to_f32(rho[x]), th = to_f32(theta[x]);
        float v[3] = {0.f, 0.f, 0.f}, in = fmaxf(fabsf(r), fabsf(th));
#pragma unroll
        for (int a = 0; a < S::D; ++a) {
            v[a] = fabsf(to_f32(u[(long long)a * cells + x]));
            in = fmaxf(in, v[a]);
        }
        if (in > 1e30f) most = __int_as_float(0x7F800000);
        static_for<4>([&](auto Sx) {
            constexpr int s = decltype(Sx)::value;
            if constexpr (shell_present<S>(s)) {
                const float ar = k.A[s] * r, bt = k.B[s] * th;
                float base = fabsf(ar + bt), parts = fabsf(ar) + fabsf(bt);
                if constexpr (s > 0) {  // the largest |c_i . u'| of the shell: of its velocities without a negative component
                    float cu = 0.f;
                    bool first = true;
                    static_for<S::Q>([&](auto I) {
                        constexpr int i = decltype(I)::value;
                        if constexpr (S::shell(i) == s && S::c(i, 0) >= 0 && S::c(i, 1) >= 0 && S::c(i, 2) >= 0) {
                            float t = 0.f;
                            static_for<3>([&](auto A) {
                                if constexpr (S::c(i, decltype(A)::value) != 0) t += v[decltype(A)::value];
                            });
                            cu = first ? t : fmaxf(cu, t);
                            first = false;
                        }
                    });
                    base = fmaf(k.C[s], cu, base);
                    parts = fmaf(k.C[s], cu, parts);
                }
                most = fmaxf(most, base);
                sum = fmaxf(sum, parts);
            }
        });
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        most = fmaxf(most, __shfl_xor_sync(kFull, most, off));
        sum = fmaxf(sum, __shfl_xor_sync(kFull, sum, off));
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMax(maxbits, __float_as_uint(most));
        atomicMax(maxbits + 1, __float_as_uint(sum));
    }
}

// Largest |g_i^eq / f*_i| of the initial fields, as float bits for atomicMax (non-negative floats
// order like their bit patterns).
template <class S>
__global__ void k_init_maxabs(const double *__restrict__ rho, const double *__restrict__ u,
                              const double *__restrict__ theta, long long cells, SetConsts k,
                              unsigned int *__restrict__ maxbits) {
    unsigned long long mb = 0;  // of the magnitudes' bits, which order like the magnitudes
    for (long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x; x < cells; x += (long long)gridDim.x * blockDim.x) {
        double uu[3] = {0.0, 0.0, 0.0};
#pragma unroll
        for (int a = 0; a < S::D; ++a) uu[a] = u[(long long)a * cells + x];
        equilibrium_cell<S, 1>(rho[x], theta[x], uu, k, [&](int, double v) {
            const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFull;
            if (b <= 0x7FF0000000000000ull && b > mb) mb = b;  // (a NaN is left out, as fmaxf does)
        });
    }
    float m = (float)__longlong_as_double((long long)mb);  // the rounding keeps the order
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(kFull, m, off));
    if ((threadIdx.x & 31) == 0) atomicMax(maxbits, __float_as_uint(m));
}

// One border cell (x, y) of an open 2D grid, pulled with the entering populations of the learned
// edge and collided: ghost(e, k) gives the population entering through edge e (0: x = 0, 1:
// x = nx - 1, 2: y = 0, 3: y = ny - 1) at position k along it.  The pulls follow the fused step's
// open-edge rules and the collision is collide_cell, so the cell gets what one step run with the
// ghosts throughout gives it (a corner takes one population from each of its two edges).
// `pulled(i, xs, ys)` gives the stored value of velocity i at source cell (xs, ys) inside the grid
// (edge_fixup_cell reads it from src).
template <class S, class T, class Ghost, class Pulled>
__device__ __forceinline__ void edge_fixup_cell_from(T *__restrict__ dst, const GridDesc &gd,
                                                     const CollideCoef<typename Store<T>::C> &cf, Ghost ghost,
                                                     Pulled pulled, int x, int y) {
    static_assert(S::D == 2, "border cells of 2D grids");
    using C = typename Store<T>::C;
    const int nx = gd.nx, ny = gd.ny;
    C pull[S::Q][1], post[S::Q][1];
    static_for<S::Q>([&](auto I) {
        constexpr int i = decltype(I)::value;
        constexpr int cx = S::c(i, 0), cy = S::c(i, 1);
        const int xs = x - cx, ys = y - cy;
        C v = C(0);
        if (ys < 0 || ys >= ny) {  // enters through the bottom (c_y = +1) or top edge
            if (cx == 0) v = ghost(cy == 1 ? 2 : 3, x);
        } else if (xs < 0) {  // through the left edge
            if (cy == 0) v = ghost(0, y);
        } else if (xs >= nx) {  // through the right edge
            if (cy == 0) v = ghost(1, y);
        } else {
            v = pulled(i, xs, ys);
        }
        pull[i][0] = v;
    });
    collide_cell<S, 0>(pull, post, cf);
#pragma unroll
    for (int i = rest_static<S>() ? 1 : 0; i < S::Q; ++i) dst[(long long)i * gd.pitch + (long long)y * nx + x] = Store<T>::make(post[i][0]);
}
template <class S, class T, class Ghost>
__device__ __forceinline__ void edge_fixup_cell(const T *__restrict__ src, T *__restrict__ dst, const GridDesc &gd,
                                                const CollideCoef<typename Store<T>::C> &cf, Ghost ghost, int x,
                                                int y) {
    edge_fixup_cell_from<S, T>(dst, gd, cf, ghost, [&](int i, int xs, int ys) {
        return Store<T>::load(src[(long long)i * gd.pitch + (long long)ys * gd.nx + xs]);
    }, x, y);
}

// The border cells of an open 2D grid for one step of the learned edge, from the step's source
// state and the network's entering populations (ghost[4][L]): one thread per border cell (corners
// belong to the x-edges).  The interior cells come from the step kernel, which leaves these cells
// unwritten (OpenEdge::skip_border), so the two can run at the same time.
template <class S, class T>
__global__ void k_edge_fixup(const T *__restrict__ src, T *__restrict__ dst, GridDesc gd,
                             CollideCoef<typename Store<T>::C> cf, const typename Store<T>::C *__restrict__ ghost,
                             int L) {
    using C = typename Store<T>::C;
    const int nx = gd.nx, ny = gd.ny;
    const int nb = 2 * ny + 2 * (nx - 2);
    for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < nb; r += gridDim.x * blockDim.x) {
        int x, y;
        if (r < ny) {
            x = 0;
            y = r;
        } else if (r < 2 * ny) {
            x = nx - 1;
            y = r - ny;
        } else if (r < 2 * ny + (nx - 2)) {
            x = 1 + (r - 2 * ny);
            y = 0;
        } else {
            x = 1 + (r - 2 * ny - (nx - 2));
            y = ny - 1;
        }
        edge_fixup_cell<S, T>(src, dst, gd, cf, [&](int e, int k) -> C { return ghost[e * L + k]; }, x, y);
    }
}

// Sponge damping of a stored post-collision state: g* <- (1 - sigma(d)) g* in the frame cells.
// Applied once after init_fields so that the initial state is a post-collision state like every
// later one (the equilibrium is its own collision; the frame damping is not).
template <class S, class T>
__global__ void k_sponge_damp(T *__restrict__ g, T *__restrict__ other, GridDesc gd, int w,
                              typename Store<T>::C smax) {
    using C = typename Store<T>::C;
    const long long cells = (long long)gd.nx * gd.ny * gd.nz;
    for (long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x; x < cells; x += (long long)gridDim.x * blockDim.x) {
        const int cx = (int)(x % gd.nx);
        const long long r = x / gd.nx;
        const int cy = (int)(r % gd.ny), cz = (int)(r / gd.ny);
        const C damp = sponge_factor<C>(cx, cy, cz, gd, S::D, w, smax);
        if (damp == C(1)) continue;
#pragma unroll
        for (int i = 0; i < S::Q; ++i) {
            T *p = g + (long long)i * gd.pitch + x;
            *p = Store<T>::make(Store<T>::load(*p) * damp);
            if (rest_static<S>() && i == 0) other[x] = *p;
        }
    }
}

// Per-shell sums of one cell's stored populations in FP64: P[slot] = sum g, J[slot][a] = sum c_a g (in stored units).
// Velocities 2k-1 and 2k are opposite, so every pair gives one sum and one difference.
template <class S, class T>
__device__ __forceinline__ void shell_sums(const T *__restrict__ g, long long pitch, long long x,
                                           double (&P)[n_shells<S>()], double (&J)[n_shells<S>()][3]) {
#pragma unroll
    for (int k = 0; k < n_shells<S>(); ++k) P[k] = J[k][0] = J[k][1] = J[k][2] = -0.0;  // the first addition folds away
    P[shell_slot<S>(0)] = (double)load_elem<S, T>(g, pitch, x);
    static_for<S::Q / 2>([&](auto H) {
        constexpr int i = 1 + 2 * decltype(H)::value;
        constexpr int k = shell_slot<S>(S::shell(i));
        const double v = (double)load_elem<S, T>(g, pitch, (long long)i * pitch + x);
        const double o = (double)load_elem<S, T>(g, pitch, (long long)(i + 1) * pitch + x);
        P[k] += v + o;
        const double d = v - o;
        static_for<3>([&](auto A) {
            constexpr int a = decltype(A)::value;
            if constexpr (S::c(i, a) == 1) J[k][a] += d;
            if constexpr (S::c(i, a) == -1) J[k][a] -= d;
        });
    });
}

// Sums of values that are FP32 numbers (every storage but FP64) on the integer pipe.  With E the largest biased
// exponent among them, a value is its 24-bit mantissa, shifted left by kFixBits and right by its own distance from E: a
// 64-bit integer in units of 2^(E - 150 - kFixBits), added exactly and rounded to FP64 once.  Zeros shift out to
// nothing.  Where values are so far apart that bits of the smaller ones are shifted out (FixRange::exact is false; not in
// FP16, whose range is narrow), they add those bits in FP64 (fix_rest): a sum of small values beside large ones of another sum
// keeps the precision of an FP64 sum of its own terms.  Infinities and NaN take FP64 sums.
constexpr int kFixBits = 33, kFixBitsSq = 10;
// Whether the sums of n values stay inside their 64 bits: a value is below 2^(24 + kFixBits) in magnitude and the signed
// sum below 2^63, a square below 2^(48 + kFixBitsSq) and the unsigned sum below 2^64.
__host__ __device__ constexpr bool fix_fits(int n) {
    return n < 1 << (63 - 24 - kFixBits) && n < 1 << (64 - 48 - kFixBitsSq);
}
template <class T>
__host__ __device__ constexpr bool fixed_sums() {
    return !std::is_same<T, double>::value;
}
// Exponents by which two values may differ so that no bit is shifted out: kFixBits and the trailing zeros that the
// storage leaves in 24 bits (FP16: 11-bit mantissas, and no values further apart than 2^40).
template <class T>
__host__ __device__ constexpr int fix_spread() {
    return kFixBits + (std::is_same<T, __half>::value ? 13 : std::is_same<T, __nv_bfloat16>::value ? 16 : 0);
}
template <class T>
__host__ __device__ constexpr bool fix_always_exact() {
    return std::is_same<T, __half>::value;
}
// Magnitudes of a set of values: the largest one's bits, and those of the smallest that is not zero, less 1, of the moving
// and of the rest populations.  (Of fields with theta' in balance with rho' the rest populations are what rounding
// leaves of zero, far below the moving ones: they alone are looked at then.)
template <class T>
struct FixRange {
    unsigned most = 0, least[2] = {0xFFFFFFFFu, 0xFFFFFFFFu};
    __device__ __forceinline__ void add(unsigned bits, bool rest) {
        const unsigned a = bits & 0x7FFFFFFFu;
        most = a > most ? a : most;
        if constexpr (!fix_always_exact<T>()) least[rest] = a - 1u < least[rest] ? a - 1u : least[rest];
    }
    __device__ __forceinline__ bool finite() const { return most < 0x7F800000u; }
    __device__ __forceinline__ unsigned exponent() const { return most >> 23; }
    // whether none of the moving (rest) values loses bits
    __device__ __forceinline__ bool exact(bool rest) const {
        return fix_always_exact<T>() || least[rest] == 0xFFFFFFFFu ||
               (most >> 23) - ((least[rest] + 1u) >> 23) <= (unsigned)fix_spread<T>();
    }
};
// Zeros shift out from an exponent of 57 on.  Values that are all smaller than 2^-63 are multiplied by 2^kFixLift first,
// which makes their denormals normal numbers too; returns the factor's exponent.
constexpr int kFixLift = 100;
template <class T, int N, int Q>
__device__ __forceinline__ int fix_lift(unsigned (&b)[N][Q], FixRange<T> &range) {
    if (fix_always_exact<T>() || range.most >= 64u << 23) return 0;
    range = FixRange<T>();
#pragma unroll
    for (int c = 0; c < N; ++c)
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            b[c][i] = __float_as_uint(__uint_as_float(b[c][i]) * 0x1p100f);
            range.add(b[c][i], i == 0);
        }
    return kFixLift;
}
__device__ __forceinline__ int fix_shift(unsigned bits, unsigned E) {
    const int s = (int)(E - ((bits >> 23) & 0xFFu));
    return s < 63 ? s : 63;
}
__device__ __forceinline__ long long fix_value(unsigned bits, int shift) {
    const long long m = (long long)(((unsigned long long)((bits & 0x7FFFFFu) | 0x800000u) << kFixBits) >> shift);
    const long long sign = (int)bits >> 31;
    return (m ^ sign) - sign;
}
// The part of a value that fix_value shifts out (exact in FP32), by exponent E and lift of its set.
__device__ __forceinline__ double fix_rest(float value, unsigned E, int lift) {
    if (lift) value *= 0x1p100f;
    const unsigned bits = __float_as_uint(value);
    const int n = fix_shift(bits, E) - kFixBits;  // mantissa bits
    const unsigned kept = n <= 0 ? bits : n < 24 ? bits & ~((1u << n) - 1u) : 0u;
    const double rest = (double)(value - __uint_as_float(kept));
    return lift ? rest * 0x1p-100 : rest;
}
// Its square, in units of 2^(2 (E - 150) - kFixBitsSq); squares add up, so what small ones lose (2^-58 of the largest)
// is less than an FP64 sum's rounding.
__device__ __forceinline__ unsigned long long fix_square(unsigned bits, int shift) {
    const unsigned m = (bits & 0x7FFFFFu) | 0x800000u;
    const int s = 2 * shift;
    return (((unsigned long long)m * m) << kFixBitsSq) >> (s < 63 ? s : 63);
}
// v 2^e as FP64, v rounded once to nearest even: two dozen integer instructions, which cost less than the one
// conversion of the FP64 pipe (2 against 128 lanes per clock).
template <class I>
__device__ __forceinline__ double fix_double(I v, int e) {
    bool minus = false;
    if constexpr (std::is_signed<I>::value) minus = v < 0;
    const unsigned long long u = minus ? 0ull - (unsigned long long)v : (unsigned long long)v;
    const int n = __clzll((long long)u);
    const unsigned long long m = u << (n & 63);  // the leading bit on top
    unsigned long long q = m >> 11;
    q += (((unsigned)m & 0x7FFu) + 0x3FFu + ((unsigned)q & 1u)) >> 11;  // (a carry out of 53 bits raises the exponent)
    const int hi = (int)(q >> 32) + ((1023 + 63 - 1 - n + e) << 20);
    return u == 0 ? 0.0 : __hiloint2double(minus ? hi | (int)0x80000000 : hi, (int)(unsigned)q);
}

// Per-cell moments (Sec. 4 discrete moments, Sec. 5 temperature) in FP64.
// D3Q7 384^3 FP32: 2.89 ms with FP64 sums and conversions, 0.97 ms with integer ones (0.57 at the copy rate);
// D3Q19 256^3: 2.44 -> 0.53 ms.
template <class S, class T>
__global__ void k_moments(const T *__restrict__ g, long long cells, long long pitch, SetConsts k, double *__restrict__ rho,
                          double *__restrict__ u, double *__restrict__ theta) {
    constexpr bool scaled = Store<T>::scaled;
    constexpr int NS = n_shells<S>(), D = S::D;
    static_assert(fix_fits(S::Q), "integer sums of a cell");
    for (long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x; x < cells; x += (long long)gridDim.x * blockDim.x) {
        // shell sums; where the storage is not scaled their total and the momentum over all shells, else the
        // momentum of each
        constexpr int NJ = scaled ? NS : 1;
        double P[NS], J[NJ][3] = {}, total = 0.0;
        bool done = false;
        if constexpr (fixed_sums<T>()) {
            unsigned b[1][S::Q];
            FixRange<T> range;
            static_for<S::Q>([&](auto I) {
                constexpr int i = decltype(I)::value;
                b[0][i] = __float_as_uint((float)load_elem<S, T>(g, pitch, (long long)i * pitch + x));
                range.add(b[0][i], i == 0);
            });
            if (range.most == 0) {
                done = true;
#pragma unroll
                for (int s = 0; s < NS; ++s) P[s] = 0.0;
            } else if (range.finite()) {
                done = true;
                const int lift = fix_lift<T>(b, range);
                const unsigned E = range.exponent();
                long long p[NS], j[NJ][3], all = 0;
#pragma unroll
                for (int s = 0; s < NS; ++s) p[s] = 0;
#pragma unroll
                for (int s = 0; s < NJ; ++s) j[s][0] = j[s][1] = j[s][2] = 0;
                static_for<S::Q>([&](auto I) {
                    constexpr int i = decltype(I)::value;
                    constexpr int s = shell_slot<S>(S::shell(i)), sj = scaled ? s : 0;
                    const long long v = fix_value(b[0][i], fix_shift(b[0][i], E));
                    p[s] += v;
                    static_for<D>([&](auto A) {
                        constexpr int a = decltype(A)::value;
                        if constexpr (S::c(i, a) == 1) j[sj][a] += v;
                        if constexpr (S::c(i, a) == -1) j[sj][a] -= v;
                    });
                });
                const int e = (int)E - 150 - kFixBits - lift;
#pragma unroll
                for (int s = 0; s < NS; ++s) {
                    all += p[s];
                    if (scaled || s > 0) P[s] = fix_double(p[s], e);
                }
                if constexpr (!scaled) total = fix_double(all, e);
                if (u) {
#pragma unroll
                    for (int s = 0; s < NJ; ++s)
#pragma unroll
                        for (int a = 0; a < D; ++a) J[s][a] = fix_double(j[s][a], e);
                }
                // and what was shifted out
                if (!range.exact(true)) {
                    const double v = fix_rest(load_elem<S, T>(g, pitch, x), E, lift);
                    if constexpr (scaled) P[0] += v;
                    else total += v;
                }
                if (!range.exact(false)) {  // (of values read again: they need no registers till here)
                    long long again = x;
                    asm volatile("" : "+l"(again));
                    double Pr[NS], Jr[NJ][3], totalr = 0.0;
#pragma unroll
                    for (int s = 0; s < NS; ++s) Pr[s] = 0.0;
#pragma unroll
                    for (int s = 0; s < NJ; ++s) Jr[s][0] = Jr[s][1] = Jr[s][2] = 0.0;
                    static_for<S::Q - 1>([&](auto I) {
                        constexpr int i = 1 + decltype(I)::value;
                        constexpr int s = shell_slot<S>(S::shell(i)), sj = scaled ? s : 0;
                        const double v = fix_rest(load_elem<S, T>(g, pitch, (long long)i * pitch + again), E, lift);
                        Pr[s] += v;
                        if constexpr (!scaled) totalr += v;
                        static_for<D>([&](auto A) {
                            constexpr int a = decltype(A)::value;
                            if constexpr (S::c(i, a) == 1) Jr[sj][a] += v;
                            if constexpr (S::c(i, a) == -1) Jr[sj][a] -= v;
                        });
                    });
#pragma unroll
                    for (int s = 1; s < NS; ++s) P[s] += Pr[s];
                    total += totalr;
#pragma unroll
                    for (int s = 0; s < NJ; ++s)
#pragma unroll
                        for (int a = 0; a < D; ++a) J[s][a] += Jr[s][a];
                }
            }
        }
        if (!done) {
            double Js[NS][3];
            shell_sums<S, T>(g, pitch, x, P, Js);
            total = -0.0;
#pragma unroll
            for (int s = 0; s < NS; ++s) total += P[s];
#pragma unroll
            for (int a = 0; a < D; ++a) {
                if constexpr (scaled) {
#pragma unroll
                    for (int s = 0; s < NS; ++s) J[s][a] = Js[s][a];
                } else {
                    J[0][a] = -0.0;
#pragma unroll
                    for (int s = 1; s < NS; ++s) J[0][a] += Js[s][a];
                }
            }
        }
        double r = scaled ? -0.0 : total, j[3] = {-0.0, -0.0, -0.0};
        static_for<4>([&](auto Sx) {
            constexpr int s = decltype(Sx)::value;
            if constexpr (shell_present<S>(s) && scaled) {
                constexpr int kk = shell_slot<S>(s);
                r = fma(P[kk], k.dec[s], r);
                if constexpr (s > 0) {  // (the rest shell has no momentum)
#pragma unroll
                    for (int a = 0; a < D; ++a) j[a] = fma(J[kk][a], k.dec[s], j[a]);
                }
            }
        });
        if (rho) rho[x] = r;
        if (u) {
#pragma unroll
            for (int a = 0; a < D; ++a) {
                const double ja = scaled ? j[a] : J[0][a];
                u[(long long)a * cells + x] = k.inv_rho0 == 1.0 ? ja : ja * k.inv_rho0;
            }
        }
        if (theta) {
            double th = -k.kR * r;
            static_for<4>([&](auto Sx) {  // (the rest shell has no energy)
                constexpr int s = decltype(Sx)::value;
                if constexpr (s > 0 && shell_present<S>(s)) th = fma(k.te[scaled ? 1 : 0][s], P[shell_slot<S>(s)], th);
            });
            theta[x] = th;
        }
    }
}

constexpr int kReduceThreads = 256;
constexpr int kReduceMax = 16;  // raw accumulators per block (<= 16, see reduce_nraw)

// Raw accumulators of a reduction, per block: for every present shell (compact slot k)
//   [k] = sum g,  [NS + k] = sum g^2,  [2 NS + k D + a] = sum c_a g   (stored units),
// and [NR - 1] = number of non-finite values.  The weights come in when the block sums are
// combined (k_reduce_final): the paper's diagnostics are linear in these shell sums.
template <class S>
__host__ __device__ constexpr int reduce_nraw() {
    return 2 * n_shells<S>() + n_shells<S>() * S::D + 1;
}

// Adds one cell in FP64: the cells of a group with infinities or NaN.
template <class S, class T>
__device__ __forceinline__ void reduce_cell(const T *__restrict__ g, long long pitch, long long x,
                                            double (&acc)[reduce_nraw<S>()]) {
    constexpr int NS = n_shells<S>(), D = S::D, NR = reduce_nraw<S>();
    static_for<S::Q>([&](auto I) {
        constexpr int i = decltype(I)::value;
        constexpr int k = shell_slot<S>(S::shell(i));
        const double v = (double)load_elem<S, T>(g, pitch, (long long)i * pitch + x);
        if (isfinite(v)) {
            acc[k] += v;
            acc[NS + k] = fma(v, v, acc[NS + k]);
            static_for<D>([&](auto A) {
                constexpr int a = decltype(A)::value;
                if constexpr (S::c(i, a) == 1) acc[2 * NS + k * D + a] += v;
                if constexpr (S::c(i, a) == -1) acc[2 * NS + k * D + a] -= v;
            });
        } else {
            acc[NR - 1] += 1.0;  // counted and left out
        }
    });
}
// Adds an FP64 state's values of N cells (one or four), `stride` apart.  A pair of opposite velocities gives a sum
// and a difference, so that momentum adds up the differences, which may be far smaller than the populations; the
// cells are added to one another before they reach the accumulator.  With one accumulator per velocity, and
// momentum from them at the end, there would be a third fewer FP64 instructions, but momentum would carry the
// roundings of the populations' sums.  (D3Q7 384^3: 3.57 ms value by value, 2.06 so.)
template <class S, int N>
__device__ __forceinline__ void reduce_group(const double *__restrict__ g, long long pitch, long long x, long long stride,
                                             double (&acc)[reduce_nraw<S>()], int &bad) {
    constexpr int NS = n_shells<S>(), D = S::D;
    auto load = [&](int i, double (&v)[N]) {
#pragma unroll
        for (int c = 0; c < N; ++c) v[c] = __ldg(g + (long long)i * pitch + x + c * stride);
#pragma unroll
        for (int c = 0; c < N; ++c)
            if ((((unsigned)__double2hiint(v[c]) >> 20) & 0x7FFu) == 0x7FFu) {  // (counted and left out)
                v[c] = 0.0;
                ++bad;
            }
    };
    auto sum = [](const double (&v)[N]) {
        if constexpr (N == 1) return v[0];
        else return (v[0] + v[1]) + (v[2] + v[3]);
    };
    double r[N];
    load(0, r);
    acc[0] += sum(r);
#pragma unroll
    for (int c = 0; c < N; ++c) acc[NS] = fma(r[c], r[c], acc[NS]);
    static_for<S::Q / 2>([&](auto H) {
        constexpr int i = 1 + 2 * decltype(H)::value;
        constexpr int k = shell_slot<S>(S::shell(i));
        double v[N], o[N], t[N];
        load(i, v);
        load(i + 1, o);
#pragma unroll
        for (int c = 0; c < N; ++c) {
            t[c] = v[c] + o[c];
            acc[NS + k] = fma(o[c], o[c], fma(v[c], v[c], acc[NS + k]));
        }
        acc[k] += sum(t);
#pragma unroll
        for (int c = 0; c < N; ++c) t[c] = v[c] - o[c];
        const double d = sum(t);
        static_for<D>([&](auto A) {
            constexpr int a = decltype(A)::value;
            if constexpr (S::c(i, a) == 1) acc[2 * NS + k * D + a] += d;
            if constexpr (S::c(i, a) == -1) acc[2 * NS + k * D + a] -= d;
        });
    });
}

// The values of four cells from cell x (zeros from `cells` on), as FP32 bits.  wide: every velocity's elements lie so
// that four of them can be read at once.
template <class S, class T>
__device__ __forceinline__ void load_group(const T *__restrict__ g, long long pitch, long long x, long long cells,
                                           bool wide, unsigned (&b)[4][S::Q]) {
    if (wide && x + 4 <= cells) {
        static_for<S::Q>([&](auto I) {
            constexpr int i = decltype(I)::value;
            const long long at = (long long)i * pitch + x;
            float v[4];
            if constexpr (std::is_same<T, Bfp16>::value) bfp_load_vec<4>(g + at, bfp_exps<S::Q>(g, pitch) + (at >> 3), v);
            else load_vec<T, 4>(g + at, v);
#pragma unroll
            for (int c = 0; c < 4; ++c) b[c][i] = __float_as_uint(v[c]);
        });
    } else {
#pragma unroll
        for (int c = 0; c < 4; ++c)
            static_for<S::Q>([&](auto I) {
                constexpr int i = decltype(I)::value;
                b[c][i] = x + c < cells ? __float_as_uint((float)load_elem<S, T>(g, pitch, (long long)i * pitch + x + c)) : 0u;
            });
    }
}

// One block's share.  FP32 and 16-bit values of a thread's kReduceGroup cells, which lie side by side (so that
// their values are of one size in a smooth field), are added as integers and reach the FP64 accumulators as one value
// per sum; the group of a shell of 12 velocities (D3Q13, D3Q19) has 48 of them.
// (D3Q7 384^3 FP32: 4.32 ms with FP64 sums of every value, 0.75 ms so, 0.24 at the copy rate; D3Q19 256^3 3.81 ->
// 0.61 ms; with cells a block's width apart 0.72 and 0.66, but 1.78 and 3.19 where a pulse falls off, now 0.47 and 0.64).
constexpr int kReduceGroup = 4;
template <class S>
__host__ __device__ constexpr int most_in_shell() {
    int most = 0;
    for (int s = 0; s < 4; ++s) {
        int n = 0;
        for (int i = 0; i < S::Q; ++i) n += S::shell(i) == s ? 1 : 0;
        most = n > most ? n : most;
    }
    return most;
}
// Blocks per SM: the launch has three (reduce_blocks) where their registers fit.
template <class S>
__host__ __device__ constexpr int reduce_min_blocks() {
    return S::Q <= 9 ? 3 : S::Q <= 13 ? 2 : 1;
}
template <class S, class T>
__global__ void __launch_bounds__(kReduceThreads, reduce_min_blocks<S>())
    k_reduce_partial(const T *__restrict__ g, long long cells, long long pitch, double *__restrict__ partial) {
    constexpr int NS = n_shells<S>(), D = S::D, NR = reduce_nraw<S>(), G = kReduceGroup;
    static_assert(NR <= kReduceMax, "raw accumulators do not fit");
    static_assert(G == 4 && fix_fits(G * most_in_shell<S>()), "integer sums of a group's shell");
    double acc[NR];
#pragma unroll
    for (int v = 0; v < NR; ++v) acc[v] = 0.0;
    if constexpr (fixed_sums<T>()) {
        const long long span = (long long)kReduceThreads * G;
        const bool wide = pitch % 4 == 0 && reinterpret_cast<unsigned long long>(g) % (4 * sizeof(T)) == 0;
        for (long long x0 = (long long)blockIdx.x * span + G * threadIdx.x; x0 < cells; x0 += (long long)gridDim.x * span) {
            unsigned b[G][S::Q];
            load_group<S, T>(g, pitch, x0, cells, wide, b);
            FixRange<T> range;
#pragma unroll
            for (int c = 0; c < G; ++c)
#pragma unroll
                for (int i = 0; i < S::Q; ++i) range.add(b[c][i], i == 0);
            if (range.most == 0) continue;  // (zeros add nothing)
            if (!range.finite()) {
#pragma unroll 1
                for (long long x = x0; x < x0 + G && x < cells; ++x) reduce_cell<S, T>(g, pitch, x, acc);
                continue;
            }
            const int lift = fix_lift<T>(b, range);
            const unsigned E = range.exponent();
            long long p[NS], j[NS][3];
            unsigned long long q[NS];
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                q[s] = 0;
                p[s] = j[s][0] = j[s][1] = j[s][2] = 0;
            }
#pragma unroll
            for (int c = 0; c < G; ++c) {
                static_for<S::Q>([&](auto I) {
                    constexpr int i = decltype(I)::value;
                    constexpr int s = shell_slot<S>(S::shell(i));
                    const int shift = fix_shift(b[c][i], E);
                    const long long v = fix_value(b[c][i], shift);
                    p[s] += v;
                    q[s] += fix_square(b[c][i], shift);
                    static_for<D>([&](auto A) {
                        constexpr int a = decltype(A)::value;
                        if constexpr (S::c(i, a) == 1) j[s][a] += v;
                        if constexpr (S::c(i, a) == -1) j[s][a] -= v;
                    });
                });
            }
            const int e = (int)E - 150 - lift;
            static_for<NS>([&](auto Kx) {
                constexpr int k = decltype(Kx)::value;
                acc[k] += fix_double(p[k], e - kFixBits);
                acc[NS + k] += fix_double(q[k], 2 * e - kFixBitsSq);
                if constexpr (k > 0) {
#pragma unroll
                    for (int a = 0; a < D; ++a) acc[2 * NS + k * D + a] += fix_double(j[k][a], e - kFixBits);
                }
            });
            // and what was shifted out, of values read again
            if (!range.exact(true)) {
#pragma unroll 1
                for (long long x = x0; x < x0 + G && x < cells; ++x) acc[0] += fix_rest(load_elem<S, T>(g, pitch, x), E, lift);
            }
            if (!range.exact(false)) {
#pragma unroll 1
                for (long long x = x0; x < x0 + G && x < cells; ++x) {
                    static_for<S::Q - 1>([&](auto I) {
                        constexpr int i = 1 + decltype(I)::value;
                        constexpr int s = shell_slot<S>(S::shell(i));
                        const double v = fix_rest(load_elem<S, T>(g, pitch, (long long)i * pitch + x), E, lift);
                        acc[s] += v;
                        static_for<D>([&](auto A) {
                            constexpr int a = decltype(A)::value;
                            if constexpr (S::c(i, a) == 1) acc[2 * NS + s * D + a] += v;
                            if constexpr (S::c(i, a) == -1) acc[2 * NS + s * D + a] -= v;
                        });
                    });
                }
            }
        }
    } else {
        const long long stride = (long long)gridDim.x * kReduceThreads;
        int bad = 0;
        long long x = (long long)blockIdx.x * kReduceThreads + threadIdx.x;
        for (; x + (G - 1) * stride < cells; x += G * stride) reduce_group<S, G>(g, pitch, x, stride, acc, bad);
        for (; x < cells; x += stride) reduce_group<S, 1>(g, pitch, x, stride, acc, bad);
        acc[NR - 1] = (double)bad;
    }
    __shared__ double sh[kReduceThreads / 32][NR];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int v = 0; v < NR; ++v) {
        double a = acc[v];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) a += __shfl_down_sync(kFull, a, off);
        if (lane == 0) sh[warp][v] = a;
    }
    __syncthreads();
    if (threadIdx.x < NR) {
        double a = 0.0;
        for (int w = 0; w < kReduceThreads / 32; ++w) a += sh[w][threadIdx.x];
        partial[(long long)blockIdx.x * kReduceMax + threadIdx.x] = a;
    }
}

// How the raw block sums combine into the D + 4 diagnostics of lee_lbm_reduce:
//   sum rho' = sum_k dec_k P_k, sum j_a = sum_k dec_k J_ka, energy moment = sum_k ew_k dec_k P_k,
//   weighted energy = sum_k dec_k^2 Sq_k / f*_k, non-finite count (dec_k = 1 unless the storage
//   is scaled).
struct ReduceCombine {
    int D, ns, nraw;
    double dec[4], ew[4], f[4];  // per compact slot
};

// Ordered sum of the block partials (one warp per raw value) and the combination above; one
// block of 32 * nraw threads.
__global__ void k_reduce_final(const double *__restrict__ partial, int nblocks, ReduceCombine c, double *__restrict__ out);

// FP64 [q][cells] <-> storage (checkpoint export / import).
template <class S, class T>
__global__ void k_export(const T *__restrict__ g, long long cells, long long pitch, SetConsts k, double *__restrict__ out) {
    constexpr bool scaled = Store<T>::scaled;
    for (long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x; x < cells; x += (long long)gridDim.x * blockDim.x) {
        static_for<S::Q>([&](auto I) {
            constexpr int i = decltype(I)::value;
            out[(long long)i * cells + x] = decode<S>((double)load_elem<S, T>(g, pitch, (long long)i * pitch + x), i, k, scaled);
        });
    }
}

template <class S, class T>
__global__ void k_import(const double *__restrict__ in, long long cells, long long pitch, SetConsts k, T *__restrict__ g,
                         T *__restrict__ other) {
    constexpr bool scaled = Store<T>::scaled;
    for (long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x; x < cells; x += (long long)gridDim.x * blockDim.x) {
        static_for<S::Q>([&](auto I) {
            constexpr int i = decltype(I)::value;
            constexpr int s = S::shell(i);
            const double v = in[(long long)i * cells + x];
            const double st = scaled ? v * k.enc[s] : v;
            const T e = Store<T>::make((typename Store<T>::C)st);
            g[(long long)i * pitch + x] = e;
            if (rest_static<S>() && i == 0) other[x] = e;
        });
    }
}

// ---------------------------------------------------------------------------------------------
// slab halos: a grid that is one slab of a periodic domain cut along its last axis
// ---------------------------------------------------------------------------------------------
// A population crosses the cut if its velocity moves along the last axis a = D - 1.  Messages hold
// one plane per crossing velocity, in the library's velocity order.
template <class S>
__host__ __device__ constexpr int slab_crossing() {
    int n = 0;
    for (int i = 0; i < S::Q; ++i) n += S::c(i, S::D - 1) == 1 ? 1 : 0;
    return n;
}
// Position of velocity i among the crossing velocities with c_a = sign.
template <class S>
__host__ __device__ constexpr int slab_slot(int i, int sign) {
    int n = 0;
    for (int j = 0; j < i; ++j) n += S::c(j, S::D - 1) == sign ? 1 : 0;
    return n;
}

// g points at the first owned cell of a state copy (velocity arrays `pitch` apart, each with one
// halo plane before the owned planes and one after).  Pack: the populations leaving downward
// (c_a = -1) from the first owned plane into send_lo, those leaving upward (c_a = +1) from the last
// owned plane into send_hi.
template <class S, class T>
__global__ void k_slab_pack(const T *__restrict__ g, long long pitch, long long plane, int nl, T *__restrict__ send_lo,
                            T *__restrict__ send_hi) {
    constexpr int a = S::D - 1;
    for (long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x; x < plane; x += (long long)gridDim.x * blockDim.x) {
        static_for<S::Q>([&](auto I) {
            constexpr int i = decltype(I)::value;
            if constexpr (S::c(i, a) == -1)
                send_lo[(long long)slab_slot<S>(i, -1) * plane + x] = g[(long long)i * pitch + x];
            if constexpr (S::c(i, a) == 1)
                send_hi[(long long)slab_slot<S>(i, 1) * plane + x] = g[(long long)i * pitch + (long long)(nl - 1) * plane + x];
        });
    }
}
// Unpack: the populations entering from below (c_a = +1, the lower neighbour's send_hi) into the
// halo plane before the owned planes, those entering from above (c_a = -1) into the one after.
template <class S, class T>
__global__ void k_slab_unpack(T *__restrict__ g, long long pitch, long long plane, int nl, const T *__restrict__ recv_lo,
                              const T *__restrict__ recv_hi) {
    constexpr int a = S::D - 1;
    for (long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x; x < plane; x += (long long)gridDim.x * blockDim.x) {
        static_for<S::Q>([&](auto I) {
            constexpr int i = decltype(I)::value;
            if constexpr (S::c(i, a) == 1)
                g[(long long)i * pitch - plane + x] = recv_lo[(long long)slab_slot<S>(i, 1) * plane + x];
            if constexpr (S::c(i, a) == -1)
                g[(long long)i * pitch + (long long)nl * plane + x] = recv_hi[(long long)slab_slot<S>(i, -1) * plane + x];
        });
    }
}

// ---------------------------------------------------------------------------------------------
// writers of BFP16 state (bfp.cuh): every block of 8 cells is encoded together
// ---------------------------------------------------------------------------------------------
// One thread per cell with whole warps in every iteration (the loop bound is warp-uniform), so the
// 8 lanes of a block share its exponent by shuffles; cells past the grid take part as zeros and
// store nothing.  `value(i, x)` gives the FP32 value of velocity i at cell x.
template <class S, class F>
__device__ __forceinline__ void bfp_write_cells(Bfp16 *__restrict__ g, Bfp16 *__restrict__ other, long long cells,
                                                long long pitch, F &&value) {
    uint8_t *__restrict__ ex = bfp_exps<S::Q>(g, pitch);
    uint8_t *__restrict__ ox = bfp_exps<S::Q>(other, pitch);
    const long long n = (cells + kBfpBlock - 1) / kBfpBlock * kBfpBlock;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long w0 = (long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31); w0 < n; w0 += stride) {
        const long long x = w0 + (threadIdx.x & 31);
        const bool valid = x < cells;
        float v[S::Q];
        value(valid ? x : -1, v);
        static_for<S::Q>([&](auto I) {
            constexpr int i = decltype(I)::value;
            const long long e = (long long)i * pitch + x;
            const float one[1] = {v[i]};
            bfp_store_vec<1>(g + e, ex + (e >> 3), one, valid);
            if constexpr (!carried<S>(i)) bfp_store_vec<1>(other + e, ox + (e >> 3), one, valid);
        });
    }
}

// g_i = g_i^eq(rho', u', theta') (Sec. 7 initial condition), rounded to FP32 and encoded.
template <class S>
__global__ void k_init_equilibrium_bfp(const double *__restrict__ rho, const double *__restrict__ u,
                                       const double *__restrict__ theta, Bfp16 *__restrict__ g,
                                       Bfp16 *__restrict__ other, long long cells, long long pitch, SetConsts k) {
    bfp_write_cells<S>(g, other, cells, pitch, [&](long long x, float (&v)[S::Q]) {
        if (x < 0) {
#pragma unroll
            for (int i = 0; i < S::Q; ++i) v[i] = 0.f;
            return;
        }
        double uu[3] = {0.0, 0.0, 0.0};
#pragma unroll
        for (int a = 0; a < S::D; ++a) uu[a] = u[(long long)a * cells + x];
        equilibrium_cell<S, 0>(rho[x], theta[x], uu, k, [&](int i, double val) { v[i] = to_f32(val); });
    });
}

// FP64 [q][cells] -> BFP16 (resume): each value rounded to FP32, then encoded.
template <class S>
__global__ void k_import_bfp(const double *__restrict__ in, long long cells, long long pitch, Bfp16 *__restrict__ g,
                             Bfp16 *__restrict__ other) {
    bfp_write_cells<S>(g, other, cells, pitch, [&](long long x, float (&v)[S::Q]) {
#pragma unroll
        for (int i = 0; i < S::Q; ++i) v[i] = x < 0 ? 0.f : (float)in[(long long)i * cells + x];
    });
}

// Sponge damping of a stored BFP16 state (after init_fields): decoded, damped as in the FP32
// kernel, re-encoded (in place: each warp reads its blocks before it writes them).
template <class S>
__global__ void k_sponge_damp_bfp(Bfp16 *__restrict__ g, Bfp16 *__restrict__ other, GridDesc gd, int w, float smax) {
    const long long cells = (long long)gd.nx * gd.ny * gd.nz;
    const uint8_t *ex = bfp_exps<S::Q>(g, gd.pitch);
    bfp_write_cells<S>(g, other, cells, gd.pitch, [&](long long x, float (&v)[S::Q]) {
        if (x < 0) {
#pragma unroll
            for (int i = 0; i < S::Q; ++i) v[i] = 0.f;
            return;
        }
        const int cx = (int)(x % gd.nx);
        const long long r = x / gd.nx;
        const int cy = (int)(r % gd.ny), cz = (int)(r / gd.ny);
        const float damp = sponge_factor<float>(cx, cy, cz, gd, S::D, w, smax);
#pragma unroll
        for (int i = 0; i < S::Q; ++i) v[i] = bfp_load1(g, ex, (long long)i * gd.pitch + x) * damp;
    });
}

}  // namespace lee
