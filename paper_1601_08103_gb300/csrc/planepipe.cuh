// planepipe.cuh -- K time steps per launch on periodic 3D FP32 grids of the seven-velocity sets (D3Q7 and
// diatomic D3Q7): a block marches through the planes with all K levels of the pipeline in registers.
//
// A block of T threads owns a tile of columns and rows and a segment of planes.  Thread t holds four
// adjacent cells (chunk t % C of row t / C of the tile) as an even and an odd pair (see rowpipe.cuh).
// Iteration i makes plane q_i = z0 - (K-1) + i of S(t+1) (level 1), pulled from S(t) as in the one-step
// kernel, and then plane q_i - (l-1) of S(t+l) for l = 2 .. K.  That plane pulls +-x and +-y from the same
// plane of level l-1 (made one iteration earlier), +z from plane q_i - l (two iterations earlier) and -z
// from plane q_i - l + 2 (this iteration).  +-z are the thread's own registers; +-x come by shuffle from
// the neighbouring lane, at a warp's ends through a word of shared memory; +-y come through shared memory.
// Words and rows in shared memory have two slots that alternate with the iterations.  Whatever crosses
// threads was made one iteration earlier, so one barrier per iteration orders all levels, and the reads
// of all levels can go out together.  S(t) reaches the threads through cp.async into a ring of slots,
// kPpStages - 1 planes ahead.  A warp's end lanes read their neighbours' slots too, so a slot is refilled only
// after the barrier that follows its reads.
//
// Level l is right on all but the tile's l-1 outermost rows and l outermost columns: pp_halo columns
// and K-1 rows on either side are computed and not stored, and a segment of planes costs 2 (K-1) iterations
// that store nothing.  The chunks of a row need not fill whole warps, so the host can cut any grid into
// tiles that waste little of a block (plane_pipe_cut).
//
// Every level is rounded to FP32 as a stored state is, with the operations of collide_axis_cell, so a
// launch gives the bits of K single steps.  (16-bit storage stays on the one-step kernel in 3D: it is
// rounded after every step there, whatever the calls.)
//
// What bounds it: K = 4 moves 12 bytes of DRAM per FP32 update, 0.76 of the measured copy on D3Q7 384^3 (426
// GLUPS, 256^3 373; the two-step tile of tb3d.cuh 259, one step per launch 147); a third of the computed cells are halo,
// and the warps wait for the shared-memory queue (2.5 of 8.5 cycles per issue; the barrier 0.7) with 12 warps per SM at 164
// registers, issue slots 35 % busy (256^3).
// Refilled before the barrier, with the end lanes' words copied into slots of their own, 385 / 346.
// Measured on 384^3 / 256^3 with the refill before the barrier and not taken: a row of 128 columns per warp with the +-y of S(t) in
// registers (260 / 219); two rows per thread, 256 threads (352 / 345) or 384 (spills, 312 / 287); three
// levels with 512 threads (302 / 264); levels behind branches on the iteration (307 / 278); the warps' end
// words stored under a branch (315 / 283); two stages instead of three (367 / 331).
#pragma once

#include "rowpipe.cuh"

namespace lee {

constexpr int kPpThreads = 384, kPpStages = 3;

// One row of one plane of a level: the six moving populations of a thread's cells, even and odd columns.
struct PpRow {
    float2 px[2], mx[2], py[2], my[2], pz[2], mz[2];
};

// Columns on either side of a tile that are computed but not stored.
template <int K>
__host__ __device__ constexpr int pp_halo() {
    return (K + 3) / 4 * 4;
}

// Shared memory: +-y of levels 1 .. K-1 and the warps' end columns of these levels (two slots each; one
// word that nobody reads), and the ring of planes on their way.
template <int K>
__host__ __device__ constexpr int pp_level_bytes() {
    return (K - 1) * 2 * 2 * kPpThreads * (int)sizeof(float4);
}
template <int K>
__host__ __device__ constexpr int pp_edge_bytes() {
    return (K - 1) * 2 * (kPpThreads / 32) * 2 * (int)sizeof(float) + 16;
}
template <int K>
__host__ __device__ constexpr int pp_smem_bytes() {
    return pp_level_bytes<K>() + pp_edge_bytes<K>() + kPpStages * 6 * kPpThreads * (int)sizeof(float4);
}

// A cut of the grid: C chunks per tile row (halo included), `width` columns and `height` rows stored per
// tile, HZ planes per segment.
struct PpCut {
    int C, width, height, HZ;
};

// The cut that takes the fewest iterations on `capacity` resident blocks (waves x planes marched), over
// the numbers of strips and segments a grid can be cut into.
inline PpCut plane_pipe_cut(int K, int halo, int nx, int ny, int nz, int capacity) {
    PpCut best{0, 0, 0, 0};
    double least = 0.0;
    // at most this many chunks leave a tile the rows that it needs around one that is stored
    const int most = kPpThreads / (2 * (K - 1) + 1), n0 = (nx + 4 * most - 2 * halo - 1) / (4 * most - 2 * halo);
    for (int n = n0; n < n0 + 64; ++n) {
        const int width = ((nx + n - 1) / n + 3) / 4 * 4, C = (width + 2 * halo) / 4;
        const int height = kPpThreads / C - 2 * (K - 1);
        if (height < 1) continue;  // (the first width, rounded up to whole chunks)
        const long long tiles = (long long)((nx + width - 1) / width) * ((ny + height - 1) / height);
        for (int m = 1; m <= 64 && m <= nz; ++m) {
            const int HZ = (nz + m - 1) / m, segs = (nz + HZ - 1) / HZ;
            const long long waves = (tiles * segs + capacity - 1) / capacity;
            const double cost = (double)waves * (HZ + 1.5 * (K - 1));
            if (best.C == 0 || cost < 0.999 * least) {
                least = cost;
                best = PpCut{C, width, height, HZ};
            }
        }
        if (width == 4) break;
    }
    return best;
}

// kRagged: nx is not a multiple of 4, and the four cells of a thread are copied and stored one by one.
template <int K, bool kRagged>
__global__ void __launch_bounds__(kPpThreads, 1) k_plane_pipe(const float *__restrict__ src, float *__restrict__ dst,
                                                              int nx, int ny, int nz, long long pitch, PpCut cut,
                                                              float w) {
    static_assert(K >= 2, "levels between S(t) and the output");
    constexpr int T = kPpThreads, kWarps = T / 32, kHalo = pp_halo<K>();
    extern __shared__ __align__(16) char pp_smem[];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int tile_row = t / cut.C, chunk = t - tile_row * cut.C;
    // +y (v = 0) and -y (v = 1) of thread `of` at level l, one float4 (E, O)
    auto cell = [&](int l, int slot, int v, int of) -> float4 * {
        return reinterpret_cast<float4 *>(pp_smem) + (((l - 1) * 2 + slot) * 2 + v) * T + of;
    };
    // a warp's last +x (side 0) and first -x (side 1) of level l
    auto edge = [&](int l, int slot, int of, int side) -> float * {
        return reinterpret_cast<float *>(pp_smem + pp_level_bytes<K>()) + (((l - 1) * 2 + slot) * kWarps + of) * 2 + side;
    };
    float *spare = reinterpret_cast<float *>(pp_smem + pp_level_bytes<K>() + pp_edge_bytes<K>()) - 4;
    const int x0 = blockIdx.x * cut.width, y0 = blockIdx.y * cut.height, z0 = blockIdx.z * cut.HZ;
    const int planes = min(cut.HZ, nz - z0);
    const int col = x0 - kHalo + 4 * chunk, y = y0 - (K - 1) + tile_row;
    const bool live = chunk * 4 >= kHalo && chunk * 4 < kHalo + cut.width && col < nx && tile_row >= K - 1 &&
                      tile_row < K - 1 + cut.height && y < ny;
    // the threads next to this one in y and x (itself where the tile ends) and the warps next to its own
    const int below = t >= cut.C ? t - cut.C : t, above = t + cut.C < T ? t + cut.C : t;
    const int before = t > 0 ? t - 1 : 0, after = t + 1 < T ? t + 1 : t;
    const int warp_before = warp > 0 ? warp - 1 : 0, warp_after = warp + 1 < kWarps ? warp + 1 : warp;
    const bool end_lane = lane == 0 || lane == 31;
    auto wrap = [](int v, int n) {
        v %= n;
        return v < 0 ? v + n : v;
    };
    const int plane = nx * ny;
    // the thread's four cells in rows y-1, y and y+1 of a plane
    const int xa = wrap(col, nx);
    const int row_of[3] = {wrap(y - 1, ny) * nx + xa, wrap(y, ny) * nx + xa, wrap(y + 1, ny) * nx + xa};
    int off[4];  // the thread's cells from its first one
#pragma unroll
    for (int e = 0; e < 4; ++e) off[e] = wrap(col + e, nx) - xa;
    // first elements of planes q-1, q, q+1 of S(t); z: plane q+1
    struct At {
        int m, o, p, z;
    };
    auto next_plane = [&](At &a) {
        a.m = a.o;
        a.o = a.p;
        a.p += plane;
        if (++a.z == nz) {
            a.z = 0;
            a.p = 0;
        }
    };
    At far;
    far.m = wrap(z0 - K, nz) * plane;
    far.o = wrap(z0 - K + 1, nz) * plane;
    far.z = wrap(z0 - K + 2, nz);
    far.p = far.z * plane;
    constexpr int kRow = T * (int)sizeof(float4), kStage = 6 * kRow;
    char *ring = pp_smem + pp_level_bytes<K>() + pp_edge_bytes<K>();
    const unsigned ring_at = (unsigned)__cvta_generic_to_shared(ring);
    int slot = 0, free_slot = kPpStages - 1;  // the plane to use now; the slot to fetch into
    auto fetch = [&](int to) {
#pragma unroll
        for (int v = 0; v < 6; ++v) {  // velocity v + 1: +x -x +y -y +z -z, before the +-x shift
            const int from = (v == 4 ? far.m : v == 5 ? far.p : far.o) + row_of[v == 2 ? 0 : v == 3 ? 2 : 1];
            const unsigned at = ring_at + to * kStage + v * kRow + t * 16;
            if constexpr (kRagged) {
#pragma unroll
                for (int e = 0; e < 4; ++e) copy_async<4>(at + 4 * e, src + (v + 1) * pitch + (from + off[e]));
            } else {
                copy_async<16>(at, src + (v + 1) * pitch + from);
            }
        }
        next_plane(far);
    };
    auto take = [&](int v, int of) {
        return *reinterpret_cast<const float4 *>(ring + slot * kStage + v * kRow + of * 16);
    };

    // handed on by levels 1 .. K-1: +-x of the last plane, +z of the last two (slot = parity of the iteration)
    float2 hx[K][2][4], hz[K][2][2];
    const float2 wp = splat2(w), m3 = splat2(-3.0f);
    // the collision of the pulls a, b, c, d, e, f (+x -x +y -y +z -z)
    auto collide = [&](const float2 (&a)[2], const float2 (&b)[2], const float2 (&c)[2], const float2 (&d)[2],
                       const float2 (&e)[2], const float2 (&f)[2], PpRow &r) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float2 s0 = __fadd2_rn(a[h], b[h]), s1 = __fadd2_rn(c[h], d[h]), s2 = __fadd2_rn(e[h], f[h]);
            const float2 sum = __fadd2_rn(__fadd2_rn(s0, s1), s2);
            const float2 t0 = __ffma2_rn(m3, s0, sum), t1 = __ffma2_rn(m3, s1, sum), t2 = __ffma2_rn(m3, s2, sum);
            r.px[h] = __ffma2_rn(wp, t0, a[h]);
            r.mx[h] = __ffma2_rn(wp, t0, b[h]);
            r.py[h] = __ffma2_rn(wp, t1, c[h]);
            r.my[h] = __ffma2_rn(wp, t1, d[h]);
            r.pz[h] = __ffma2_rn(wp, t2, e[h]);
            r.mz[h] = __ffma2_rn(wp, t2, f[h]);
        }
    };
    // +-x pulls from the even and odd pairs and the outer neighbours' cells
    auto shift = [&](float2 pe, float2 po, float2 me, float2 mo, float left, float right, float2 (&a)[2], float2 (&b)[2]) {
        a[0] = make_float2(left, po.x);
        a[1] = pe;
        b[0] = mo;
        b[1] = make_float2(me.y, right);
    };
    // level 1
    auto first = [&](PpRow &r) {
        float2 g[6][2];
#pragma unroll
        for (int v = 0; v < 6; ++v) {
            const float4 q = take(v, t);
            g[v][0] = make_float2(q.x, q.z);
            g[v][1] = make_float2(q.y, q.w);
        }
        float left = __shfl_up_sync(kFull, g[0][1].y, 1), right = __shfl_down_sync(kFull, g[1][0].x, 1);
        // a warp's ends: the next thread's cells, in its slot of the ring (the barrier has passed)
        const float4 q = take(lane == 31 ? 1 : 0, lane == 31 ? after : before);
        left = lane == 0 ? q.w : left;
        right = lane == 31 ? q.x : right;
        float2 a[2], b[2];
        shift(g[0][0], g[0][1], g[1][0], g[1][1], left, right, a, b);
        collide(a, b, g[2], g[3], g[4], g[5], r);
    };
    // level l as made now, kept for the next iterations
    auto hand_on = [&](auto L, auto P, const PpRow &r) {
        constexpr int l = decltype(L)::value, p = decltype(P)::value;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            hx[l][p][h] = r.px[h];
            hx[l][p][2 + h] = r.mx[h];
            hz[l][p][h] = r.pz[h];
        }
        *(end_lane ? edge(l, p, warp, lane == 0) : spare) = lane == 0 ? r.mx[0].x : r.px[1].y;  // (no branch)
        *cell(l, p, 0, t) = make_float4(r.py[0].x, r.py[0].y, r.py[1].x, r.py[1].y);
        *cell(l, p, 1, t) = make_float4(r.my[0].x, r.my[0].y, r.my[1].x, r.my[1].y);
    };
    // level l + 1 from level l, made now as r; r becomes level l + 1
    auto advance = [&](auto L, auto P, PpRow &r) {
        constexpr int l = decltype(L)::value, p = decltype(P)::value, q = p ^ 1;
        const float4 lo = *cell(l, q, 0, below), hi = *cell(l, q, 1, above);
        const float2 c[2] = {make_float2(lo.x, lo.y), make_float2(lo.z, lo.w)};
        const float2 d[2] = {make_float2(hi.x, hi.y), make_float2(hi.z, hi.w)};
        const float2 po = hx[l][q][1], me = hx[l][q][2];
        float left = __shfl_up_sync(kFull, po.y, 1), right = __shfl_down_sync(kFull, me.x, 1);
        const float end = *edge(l, q, lane == 31 ? warp_after : warp_before, lane == 31);
        left = lane == 0 ? end : left;
        right = lane == 31 ? end : right;
        float2 a[2], b[2];
        shift(hx[l][q][0], po, me, hx[l][q][3], left, right, a, b);
        const float2 e[2] = {hz[l][p][0], hz[l][p][1]}, f[2] = {r.mz[0], r.mz[1]};
        hand_on(L, P, r);
        collide(a, b, c, d, e, f, r);
    };

#pragma unroll
    for (int k = 0; k < kPpStages - 1; ++k) {
        fetch(k);
        copy_commit();
    }
    int to = (z0 - 2 * (K - 1)) * plane + y * nx + col;  // where the next iteration stores, if it does
    // Iteration i makes levels 1 .. i / 2 + 1; kAll: every level, so that it is straight code.
    auto iteration = [&](int i, auto P, auto kAll) {
        constexpr bool all = decltype(kAll)::value;
        copy_wait<kPpStages - 2>();
        // The plane, and levels 1 .. K-1 of the iteration before, are visible; their other slots are free, and so is
        // the ring slot of the plane before, which the neighbouring warps read too (first): it is fetched into from here.
        __syncthreads();
        fetch(free_slot);  // (the last ones of a segment are not used)
        copy_commit();
        PpRow r;
        first(r);
        static_for<K - 1>([&](auto Lx) {
            constexpr std::integral_constant<int, 1 + decltype(Lx)::value> L{};
            if (all || i >= 2 * L.value) advance(L, P, r);
            else if (i >= 2 * (L.value - 1)) hand_on(L, P, r);
        });
        if constexpr (all) {
            const float2 *from[6] = {r.px, r.mx, r.py, r.my, r.pz, r.mz};
#pragma unroll
            for (int v = 0; v < 6; ++v) {
                float *at = dst + (v + 1) * pitch + to;
                if constexpr (kRagged) {
                    const float f[4] = {from[v][0].x, from[v][1].x, from[v][0].y, from[v][1].y};
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (live && col + e < nx) at[e] = f[e];
                } else if (live) {
                    *reinterpret_cast<float4 *>(at) = make_float4(from[v][0].x, from[v][1].x, from[v][0].y, from[v][1].y);
                }
            }
        }
        free_slot = slot;
        if (++slot == kPpStages) slot = 0;
        to += plane;
    };
    for (int i = 0; i < 2 * (K - 1); i += 2) {
        iteration(i, std::integral_constant<int, 0>{}, std::false_type{});
        iteration(i + 1, std::integral_constant<int, 1>{}, std::false_type{});
    }
    for (int i = 0; i < planes; i += 2) {
        iteration(0, std::integral_constant<int, 0>{}, std::true_type{});
        if (i + 1 < planes) iteration(0, std::integral_constant<int, 1>{}, std::true_type{});
    }
    copy_wait<0>();
}

}  // namespace lee
