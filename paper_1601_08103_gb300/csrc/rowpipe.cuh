// rowpipe.cuh -- K time steps per launch on periodic 2D grids of the five-velocity sets with
// nx % 4 == 0 (FP32, FP16, BF16 and BFP16 storage): every warp marches its own strip down the rows with
// all K levels of the pipeline in registers.
//
// A warp owns a strip of 128 columns, four adjacent cells per lane, and a segment of rows.  Iteration
// i loads row r_i = y0 - K + i of S(t) (level 0), and level l = 1 .. K then computes row r_i - l of
// S(t+l).  That row pulls +x and -x from row r_i - l of level l-1 (made one iteration earlier), +y
// from row r_i - l - 1 (two iterations earlier) and -y from row r_i - l + 1 (this iteration), so a level
// hands on one row of +x, -x and two rows of +y: 16 registers.  The x neighbours come by warp
// shuffle.  Nothing passes through shared memory, there is no barrier, and warps never wait for
// one another.
//
// The lane's four columns 4L .. 4L+3 are held as an even pair E = (4L, 4L+2) and an odd pair
// O = (4L+1, 4L+3), the operands of the packed f32x2 instructions.  Moving by one column swaps E and O:
// a +x pull of the odd columns is the neighbour's E as it stands, a -x pull of the even ones the O, and
// only the other two (+x into E, -x into O) take one shuffle and one move each.  A level costs 14
// packed operations, 2 shuffles and 2 moves for four cells; the columns are interleaved again when
// they are stored.
//
// The strip's outermost columns have no neighbour on one side, so one more column on either side is
// wrong after every level: kHalo >= K columns per side are computed for nothing (with K = 8, 112 of
// 128 columns are stored).  Likewise a segment reads K rows before and after its own; level l starts
// at iteration 2l, the first at which a row that the segment needs can be made (a fully unrolled
// prologue of 2K iterations), so K (K - 1) rows of levels per segment are extra work.
//
// Rows of S(t) reach a warp through cp.async into a shared-memory ring of its own, several rows ahead.
//
// What bounds it: with K = 8 a D2Q5 FP32 update takes 4 bytes of DRAM and about 10 instructions per thread,
// 2 warps per scheduler.  Far beyond L2 FP32 is bound by DRAM (8192^2: 1611 GLUPS, 6.4 TB/s algorithmic,
// 0.95 of the measured copy), 16-bit storage by issue and instruction latency (issue slots 54 % busy; FP16
// 2126 GLUPS; BFP16 with K = 4 919).  The tile it replaced (four levels through shared memory, three barriers per
// four rows, 39 instructions per update) ran 8192^2 at 517 (FP32), 553 (FP16) and 403 (BFP16) GLUPS and
// 2048^2 FP32 at 426, against 1490 now.  Measured and not taken: loads two rows ahead into registers
// instead of the ring (8192^2 FP32 1304 GLUPS, FP16 1955: 3 of 5.6 stall cycles per issue waited for
// loads); pairs as 64-bit registers through inline PTX (1448, 2068: more moves, not fewer); hand-on slots
// with period 3, unrolled by 6 (1502, 2202, spills) or by 3 (681, 845, spills); four
// levels (811).
//
// Every level is rounded to FP32 as a stored state is, with the operations of collide_axis_cell: on
// FP32 storage a launch gives the bits of K single steps.  On 16-bit storage S(t) is widened, the
// levels in between stay FP32, and S(t+K) is rounded to the storage (with K = 8 S(t+4) too).  The shell factors of the
// scaled storages are the same for all moving velocities, so the same kernel serves every set.
#pragma once

#include "bfp.cuh"

namespace lee {

constexpr int kRpCols = 128;  // columns a warp loads
constexpr int kRpWarps = 4;   // warps per block, each on a tile of its own

// cp.async of N bytes from global to shared memory, per thread.
template <int N>
__device__ __forceinline__ void copy_async(unsigned to, const void *from) {
    if constexpr (N == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(to), "l"(from) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(to), "l"(from), "n"(N) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// Memory side of the pipelines: fetch() starts the copy of a lane's four cells of a velocity into its
// own slot of shared memory (kLane bytes at `to`; BFP16: and kLaneEx bytes at `to_ex`), take() reads
// the slot and widens it, store() rounds and stores four cells, round() is what a stored and reloaded
// value holds (not for BFP16).  kRagged: for any nx, with the four cells copied and stored one by one (their
// rows start at any element, and may wrap between them).  `idx` is an element of one velocity
// array starting at `base` (BFP16: with its exponent bytes at `ex`).  kAlign: a strip's first column is
// a multiple of it.
struct RpF32 {
    using Elem = float;
    static constexpr int kAlign = 4, kLane = 16, kLaneEx = 0;
    static constexpr bool kRagged = false;
    static __host__ __device__ const uint8_t *exps(const float *, long long) { return nullptr; }
    __device__ static __forceinline__ void fetch(unsigned to, unsigned, const float *__restrict__ base, const uint8_t *,
                                                 int idx) {
        copy_async<16>(to, base + idx);
    }
    __device__ static __forceinline__ float4 take(const char *from, const char *, int) {
        return *reinterpret_cast<const float4 *>(from);
    }
    __device__ static __forceinline__ float2 round(float2 v) { return v; }
    __device__ static __forceinline__ void store(float *__restrict__ base, uint8_t *, int idx, const float4 &v, bool live) {
        if (live) *reinterpret_cast<float4 *>(base + idx) = v;
    }
};

// FP32 at widths that are not multiples of 4.
struct RpF32Ragged : RpF32 {
    static constexpr bool kRagged = true;
};

// FP16 and BF16: S g / f*, rounded to nearest even.
template <class T>
struct Rp16 {
    using Elem = T;
    static constexpr int kAlign = 4, kLane = 8, kLaneEx = 0;
    static constexpr bool kRagged = false;
    static __host__ __device__ const uint8_t *exps(const T *, long long) { return nullptr; }
    __device__ static __forceinline__ void fetch(unsigned to, unsigned, const T *__restrict__ base, const uint8_t *, int idx) {
        copy_async<8>(to, base + idx);
    }
    __device__ static __forceinline__ float4 take(const char *from, const char *, int) {
        union {
            uint2 r;
            T e[4];
        } u;
        u.r = *reinterpret_cast<const uint2 *>(from);
        return make_float4(Store<T>::load(u.e[0]), Store<T>::load(u.e[1]), Store<T>::load(u.e[2]), Store<T>::load(u.e[3]));
    }
    __device__ static __forceinline__ float2 round(float2 v) {
        return make_float2(Store<T>::load(Store<T>::make(v.x)), Store<T>::load(Store<T>::make(v.y)));
    }
    __device__ static __forceinline__ void store(T *__restrict__ base, uint8_t *, int idx, const float4 &v, bool live) {
        const float a[4] = {v.x, v.y, v.z, v.w};
        if (live) store_vec<T, 4>(base + idx, a);
    }
};

// BFP16: a lane's four cells are half a block of 8, so lane pairs share the exponent.  A copy takes at
// least four bytes: every lane fetches the aligned word that holds its exponent byte.
template <int Q>
struct RpBfp {
    using Elem = Bfp16;
    static constexpr int kAlign = 8, kLane = 8, kLaneEx = 4;
    static constexpr bool kRagged = false;
    static __host__ __device__ const uint8_t *exps(const Bfp16 *g, long long pitch) { return bfp_exps<Q>(g, pitch); }
    __device__ static __forceinline__ void fetch(unsigned to, unsigned to_ex, const Bfp16 *__restrict__ base,
                                                 const uint8_t *__restrict__ ex, int idx) {
        copy_async<8>(to, base + idx);
        copy_async<4>(to_ex, ex + ((idx >> 3) & ~3));
    }
    __device__ static __forceinline__ float4 take(const char *from, const char *from_ex, int idx) {
        const uint2 m = *reinterpret_cast<const uint2 *>(from);
        const unsigned e = *reinterpret_cast<const unsigned *>(from_ex);
        const BfpDec k = bfp_dec((e >> (8 * ((idx >> 3) & 3))) & 255u);
        const float2 a = bfp_pair(m.x, k), b = bfp_pair(m.y, k);
        return make_float4(a.x, a.y, b.x, b.y);
    }
    __device__ static float2 round(float2 v);  // (declared only: no launch of eight on blocks)
    __device__ static __forceinline__ void store(Bfp16 *__restrict__ base, uint8_t *__restrict__ ex, int idx,
                                                 const float4 &v, bool live) {
        const float a[4] = {v.x, v.y, v.z, v.w};
        bfp_store_vec<4>(base + idx, ex + (idx >> 3), a, live);
    }
};

// Shared memory of one velocity's row for `lanes` lanes.
template <class IO>
__host__ __device__ constexpr int rp_row_bytes(int lanes = 32) {
    return lanes * (IO::kLane + IO::kLaneEx);
}

// Columns on either side of a strip that are computed but not stored.
template <int K, class IO>
__host__ __device__ constexpr int rp_halo() {
    constexpr int a = IO::kAlign;
    return (K + a - 1) / a * a;
}
template <int K, class IO>
__host__ __device__ constexpr int rp_width() {
    return kRpCols - 2 * rp_halo<K, IO>();
}

constexpr int kRpMinRows = 4;  // shortest segment

// One row of a level: the four moving populations of a lane's cells, even and odd columns.
struct RpRow {
    float2 px[2], mx[2], py[2], my[2];
};

// One tile: columns x0 .. x0 + rp_width - 1 (those below nx), rows y0 .. y0 + rows - 1, by one warp.
template <int K, class IO, int kHalo, int kStages>
__device__ __forceinline__ void rp_tile(const typename IO::Elem *__restrict__ src, typename IO::Elem *__restrict__ dst,
                                        int nx, int ny, long long pitch, float w, int x0, int y0, int rows, char *ring) {
    using Elem = typename IO::Elem;
    constexpr int kRow = rp_row_bytes<IO>(), kStage = 4 * kRow;
    static_assert(kHalo >= K && kHalo % IO::kAlign == 0 && kHalo % 4 == 0, "columns that the levels spoil");
    const int lane = threadIdx.x & 31;
    const int col = x0 - kHalo + 4 * lane;
    const bool live = 4 * lane >= kHalo && 4 * lane < kRpCols - kHalo && col < nx;
    const Elem *in[4];
    Elem *out[4];
    const uint8_t *in_ex[4];
    uint8_t *out_ex[4];
    const uint8_t *sx = IO::exps(src, pitch), *dx = IO::exps(dst, pitch);
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        in[v] = src + (v + 1) * pitch;
        out[v] = dst + (v + 1) * pitch;
        in_ex[v] = sx + (v + 1) * (pitch >> 3);
        out_ex[v] = const_cast<uint8_t *>(dx) + (v + 1) * (pitch >> 3);
    }
    auto wrap = [](int v, int n) {
        v %= n;
        return v < 0 ? v + n : v;
    };
    // the lane's cells from its first one
    int off[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) off[e] = wrap(col + e, nx) - wrap(col, nx);
    // A row of S(t) and the lane's element in it: the next to fetch and the next to use
    struct At {
        int row, idx;
    };
    auto next_row = [&](At &a) {
        a.idx += nx;
        if (++a.row == ny) {
            a.row = 0;
            a.idx -= ny * nx;
        }
    };
    At far, now;
    far.row = wrap(y0 - K, ny);
    far.idx = far.row * nx + wrap(col, nx);
    now = far;
    // Rows wait in a ring of kStages shared-memory slots, kStages - 1 of them on their way.  A lane reads
    // only what it copied itself, so its own wait is all the order that is needed; the slot that a
    // row is fetched into was read, and its values used, one iteration earlier.
    const unsigned ring_at = (unsigned)__cvta_generic_to_shared(ring);
    int slot = 0, free_slot = kStages - 1;  // the row to use now; the slot to fetch into
    auto fetch = [&](int to) {
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const unsigned at = ring_at + to * kStage + v * kRow;
            if constexpr (IO::kRagged) {
#pragma unroll
                for (int e = 0; e < 4; ++e) copy_async<4>(at + lane * IO::kLane + 4 * e, in[v] + (far.idx + off[e]));
            } else {
                IO::fetch(at + lane * IO::kLane, at + 32 * IO::kLane + lane * IO::kLaneEx, in[v], in_ex[v], far.idx);
            }
        }
        next_row(far);
    };
    auto take = [&]() {
        RpRow r;
        float2 *to[4] = {r.px, r.mx, r.py, r.my};
        copy_wait<kStages - 2>();
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const char *at = ring + slot * kStage + v * kRow;
            const float4 t = IO::take(at + lane * IO::kLane, at + 32 * IO::kLane + lane * IO::kLaneEx, now.idx);
            to[v][0] = make_float2(t.x, t.z);
            to[v][1] = make_float2(t.y, t.w);
        }
        if constexpr (IO::kAlign == 8) next_row(now);  // (only the exponents' place depends on it)
        return r;
    };
    auto turn = [&]() {
        free_slot = slot;
        if (++slot == kStages) slot = 0;
    };

    // What level l hands on: +x, -x of its last row and +y of its last two, slot = parity of the
    // iteration that made them.
    float2 hx[K][2][4], hy[K][2][2];
    auto hand_on = [&](auto L, auto P, const RpRow &r) {
        constexpr int l = decltype(L)::value, p = decltype(P)::value;
        hx[l][p][0] = r.px[0];
        hx[l][p][1] = r.px[1];
        hx[l][p][2] = r.mx[0];
        hx[l][p][3] = r.mx[1];
        hy[l][p][0] = r.py[0];
        hy[l][p][1] = r.py[1];
    };
    const float2 wp = splat2(w), wm = splat2(-w), m1 = splat2(-1.0f);
    // level l + 1 from level l, whose newest row is r: r becomes level l + 1's newest row.  A launch of eight
    // rounds 16-bit storage after its first four levels too, so that it gives the bits of two launches.
    auto advance = [&](auto L, auto P, RpRow &r) {
        constexpr int l = decltype(L)::value, p = decltype(P)::value;
        const float2 pe = hx[l][p ^ 1][0], po = hx[l][p ^ 1][1], me = hx[l][p ^ 1][2], mo = hx[l][p ^ 1][3];
        const float2 c[2] = {hy[l][p][0], hy[l][p][1]};
        const float left = __shfl_up_sync(kFull, po.y, 1), right = __shfl_down_sync(kFull, me.x, 1);
        const float2 a[2] = {make_float2(left, po.x), pe};
        const float2 b[2] = {mo, make_float2(me.y, right)};
        const float2 d[2] = {r.my[0], r.my[1]};
        hand_on(L, P, r);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float2 e = __ffma2_rn(m1, __fadd2_rn(a[h], b[h]), __fadd2_rn(c[h], d[h]));  // s_y - s_x
            r.px[h] = __ffma2_rn(wp, e, a[h]);
            r.mx[h] = __ffma2_rn(wp, e, b[h]);
            r.py[h] = __ffma2_rn(wm, e, c[h]);
            r.my[h] = __ffma2_rn(wm, e, d[h]);
            if constexpr (K == 8 && l + 1 == 4) {
                r.px[h] = IO::round(r.px[h]);
                r.mx[h] = IO::round(r.mx[h]);
                r.py[h] = IO::round(r.py[h]);
                r.my[h] = IO::round(r.my[h]);
            }
        }
    };

#pragma unroll
    for (int k = 0; k < kStages - 1; ++k) {
        fetch(k);
        copy_commit();
    }
    static_for<2 * K>([&](auto I) {
        constexpr int i = decltype(I)::value, p = i & 1;
        RpRow r = take();
        fetch(free_slot);
        copy_commit();
        turn();
        static_for<K>([&](auto L) {
            constexpr int l = decltype(L)::value;
            if constexpr (2 * (l + 1) <= i) {
                advance(L, std::integral_constant<int, p>{}, r);
            } else if constexpr (2 * l <= i) {
                hand_on(L, std::integral_constant<int, p>{}, r);
            }
        });
    });
    int to = y0 * nx + col;
    for (int k = 0; k < rows; k += 2) {
        static_for<2>([&](auto P) {
            constexpr int p = decltype(P)::value;
            RpRow r = take();
            if (k + p + kStages - 1 < rows) fetch(free_slot);
            copy_commit();
            turn();
            static_for<K>([&](auto L) { advance(L, P, r); });
            const bool st = live && (p == 0 || k + 1 < rows);
            const float2 *from[4] = {r.px, r.mx, r.py, r.my};
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const float4 q = make_float4(from[v][0].x, from[v][1].x, from[v][0].y, from[v][1].y);
                if constexpr (IO::kRagged) {
                    const float f[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (st && col + e < nx) out[v][to + e] = f[e];
                } else {
                    IO::store(out[v], out_ex[v], to, q, st);
                }
            }
            to += nx;
        });
    }
    copy_wait<0>();  // (a short segment fetches rows that it does not use)
}

// Slots of the ring.  FP32 states beyond L2 take four: more rows on their way make the warps drift apart
// and the halo columns and rows that neighbours share miss L2 (D2Q5 8192^2, GLUPS with 4 / 6 / 9 slots:
// 1611 / 1396 / 1391; 2048^2: 1374 / 1474 / 1509).  16-bit rows are half as long (8192^2 FP16 with 4 / 6 / 9:
// 2197 / 2228 / 2222, before the rounding of the fourth level).
constexpr long long kRpNearL2Bytes = 256LL << 20;  // both copies
constexpr int kRpStagesFar = 4, kRpStagesNear = 8, kRpStages16 = 6;

template <class IO, int kStages>
__host__ __device__ constexpr int rp_smem_bytes() {
    return kRpWarps * kStages * 4 * rp_row_bytes<IO>();
}

// Blocks per SM: 16 registers per level and about 90 more.  Eight levels leave room for two blocks of four
// warps, two warps per scheduler.
template <int K>
constexpr int rp_min_blocks() {
    return K <= 4 ? 3 : 2;
}

template <int K, class IO, int kStages>
__global__ void __launch_bounds__(32 * kRpWarps, rp_min_blocks<K>()) k_row_pipe(
    const typename IO::Elem *__restrict__ src, typename IO::Elem *__restrict__ dst, int nx, int ny, long long pitch,
    int H, int strips, int tiles, float w) {
    extern __shared__ __align__(16) char rp_smem[];
    char *ring = rp_smem + (threadIdx.x >> 5) * (kStages * 4 * rp_row_bytes<IO>());
    const int tile = blockIdx.x * kRpWarps + (threadIdx.x >> 5);
    if (tile >= tiles) return;
    const int seg = tile / strips, y0 = seg * H;
    rp_tile<K, IO, rp_halo<K, IO>(), kStages>(src, dst, nx, ny, pitch, w, (tile - seg * strips) * rp_width<K, IO>(), y0, min(H, ny - y0),
                                  ring);
}

// The same over many periodic domains: warp t works on tile tiles[t] = (domain, x0, y0) of height
// doms[domain].H.
constexpr int kRpBatchHalo = 8;  // for every K, so that one tile list serves them all
constexpr int kRpBatchWidth = kRpCols - 2 * kRpBatchHalo;
struct RpDomain {
    int nx, ny, H;
    float w;
    long long pitch, offset;
};
template <int K, int kStages>
__global__ void __launch_bounds__(32 * kRpWarps, rp_min_blocks<K>()) k_row_pipe_batched(
    const float *__restrict__ src, float *__restrict__ dst, const RpDomain *__restrict__ doms,
    const int3 *__restrict__ tiles, int count) {
    extern __shared__ __align__(16) char rp_smem[];
    char *ring = rp_smem + (threadIdx.x >> 5) * (kStages * 4 * rp_row_bytes<RpF32>());
    const int tile = blockIdx.x * kRpWarps + (threadIdx.x >> 5);
    if (tile >= count) return;
    const int3 t = tiles[tile];
    const RpDomain D = doms[t.x];
    rp_tile<K, RpF32, kRpBatchHalo, kStages>(src + D.offset, dst + D.offset, D.nx, D.ny, D.pitch, D.w, t.y, t.z, min(D.H, D.ny - t.z),
                                     ring);
}

}  // namespace lee
