// planepair.cuh -- two time steps per launch on periodic 3D FP32 grids of the sets with diagonal velocities
// (D3Q9, D3Q13, D3Q19): a block marches a tile through the planes and makes one plane of both levels per
// iteration.
//
// A block owns a tile of 64 columns and 16 rows, a warp per row and two adjacent cells per lane, and a segment of
// planes.  Iteration i makes plane q = z0 - 1 + i of S(t+1), pulled from S(t) as in the one-step kernel, and then
// plane q - 1 of S(t+2), which pulls the populations with c_z = -1 from plane q of S(t+1), those with c_z = 0
// from q - 1 and those with c_z = +1 from q - 2.  A shift in x is one shuffle; populations that move in y or up
// in z go through shared memory, the others stay with their thread.  A population is read 1 + c_z iterations after it was
// made and its array written again 3 + c_z iterations after, so with that many slots one barrier per iteration
// orders everything.  The next plane of S(t) is loaded into registers while this one's second level is made.
//
// The outermost columns have no neighbour on one side, so one more on either side is wrong after each level, and
// the outermost rows are made for S(t+1) only: 60 of 64 columns and 14 of 16 rows are stored, and a segment costs
// two iterations that store nothing.  Every operation is that of collide_shells_cell, so a launch gives the bits of
// two single steps.
//
// What bounds it: the queue of memory instructions (D3Q19: 2.3 of 10.5 cycles per issue) and the one barrier per
// plane (1.3) with 16 warps per SM at 128 registers; DRAM moves 76 bytes per D3Q19 update (152 with one step per
// launch).  us per step on 256^3, one step per launch -> now: D3Q19 393 -> 281 (0.67 of the measured copy rate),
// D3Q13 235 -> 154, D3Q9 153 -> 116; 255x249x251 (4-byte accesses) 431 -> 292, 270 -> 157.  Measured on 256^3
// (D3Q19 / D3Q13) and not taken: the cells of a lane in two rows, every access of 4 bytes, 32 columns by 16 rows and
// two blocks per SM 396 / 174 (64 columns 433 / 175; loads at their use 430 / 180; planes prefetched into L2
// 466 / 189); +z kept in registers, which spilled, 849 / 154.
#pragma once

#include "kernels.cuh"

namespace lee {

constexpr int kPairCols = 64, kPairRows = 16, kPairThreads = 32 * kPairRows;
constexpr int kPairWidth = kPairCols - 4, kPairHeight = kPairRows - 2;  // columns and rows stored
// One array of S(t+1) in shared memory: the rows of the tile and one (of zeros) before and after them, read by
// cells that are not stored.
constexpr int kPairArray = (kPairRows + 2) * kPairCols;

// Whether velocity i goes through shared memory; the number of those with c_z = cz below velocity `upto`, the slots
// of each, and the first array of that group.
template <class S>
__host__ __device__ constexpr bool pair_shared(int i) {
    return carried<S>(i) && (S::c(i, 1) != 0 || S::c(i, 2) == 1);
}
template <class S>
__host__ __device__ constexpr int pair_count(int cz, int upto = S::Q) {
    int n = 0;
    for (int i = 0; i < upto; ++i) n += pair_shared<S>(i) && S::c(i, 2) == cz ? 1 : 0;
    return n;
}
__host__ __device__ constexpr int pair_slots(int cz) { return 3 + cz; }
template <class S>
__host__ __device__ constexpr int pair_base(int cz) {
    int n = 0;
    for (int k = -1; k < cz; ++k) n += pair_count<S>(k) * pair_slots(k);
    return n;
}
template <class S>
__host__ __device__ constexpr int pair_smem_bytes() {
    return pair_base<S>(2) * kPairArray * (int)sizeof(float);
}

// Planes per segment for the fewest iterations on `capacity` resident blocks (waves x planes marched), or 0 where
// less than kPairLeast of the cells that the blocks' slots make by then are the grid's: narrow or thin grids,
// which run faster one step at a time (D3Q19, two steps against one: 256^3 with 0.77 of them 1.40 times as fast,
// 320x24x320 with 0.66 1.31, 24x320x320 with 0.32 1.03).
constexpr double kPairLeast = 0.4;
inline int plane_pair_segment(int nx, int ny, int nz, int capacity) {
    const long long tiles = (long long)((nx + kPairWidth - 1) / kPairWidth) * ((ny + kPairHeight - 1) / kPairHeight);
    int best = nz;
    double least = 0.0;
    for (int m = 1; m <= 256 && m <= nz; ++m) {
        const int HZ = (nz + m - 1) / m, segs = (nz + HZ - 1) / HZ;
        const double cost = (double)((tiles * segs + capacity - 1) / capacity) * (HZ + 2);
        if (m == 1 || cost < 0.999 * least) {
            least = cost;
            best = HZ;
        }
    }
    const double made = least * capacity * kPairWidth * kPairHeight;
    return (double)nx * ny * nz < kPairLeast * made ? 0 : best;
}

// kRagged: nx is odd, and the two cells of a lane are loaded and stored one by one.
template <class S, bool kRagged>
__global__ void __launch_bounds__(kPairThreads, 1) k_plane_pair(const float *__restrict__ src, float *__restrict__ dst,
                                                                int nx, int ny, int nz, long long pitch, int HZ,
                                                                CollideCoef<float> cf) {
    extern __shared__ __align__(16) float pair_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int x0 = blockIdx.x * kPairWidth, y0 = blockIdx.y * kPairHeight, z0 = blockIdx.z * HZ;
    const int planes = min(HZ, nz - z0);
    auto wrap = [](int v, int n) {
        v %= n;
        return v < 0 ? v + n : v;
    };
    const int x = x0 - 2 + 2 * lane, y = y0 - 1 + warp;
    const int col = wrap(x, nx), step = wrap(x + 1, nx) - col;  // the lane's first cell, and from it to its second
    // rows that a cell pulls from, by 1 + c_y
    const int row[3] = {wrap(y + 1, ny) * nx, wrap(y, ny) * nx, wrap(y - 1, ny) * nx};
    const bool live = lane >= 1 && lane <= 30 && x < nx && warp >= 1 && warp <= kPairHeight && y < ny;

    for (int k = threadIdx.x; k < pair_smem_bytes<S>() / (int)sizeof(float4); k += kPairThreads)
        reinterpret_cast<float4 *>(pair_smem)[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();

    const int plane = nx * ny;
    int zp = wrap(z0, nz);
    int from[3] = {zp * plane, wrap(z0 - 1, nz) * plane, wrap(z0 - 2, nz) * plane};  // planes q + 1, q, q - 1
    float *const mine = pair_smem + (1 + warp) * kPairCols + 2 * lane;
    float2 next[S::Q];  // the next plane's sources, before the shift in x
    auto fetch = [&] {
        static_for_carried<S>([&](auto I) {
            constexpr int v = decltype(I)::value;
            int o = from[1 + S::c(v, 2)] + row[1 + S::c(v, 1)] + col;
            asm volatile("" : "+r"(o));  // (else every population gets a pointer of its own, and they spill)
            const float *p = src + v * pitch + o;
            if constexpr (kRagged) next[v] = make_float2(__ldg(p), __ldg(p + step));
            else next[v] = __ldg(reinterpret_cast<const float2 *>(p));
        });
        from[2] = from[1];
        from[1] = from[0];
        if (++zp == nz) zp = 0;
        from[0] = zp * plane;
    };
    // the lane's cells pulled along c_x from the sources in their own columns
    auto shifted = [&](auto CX, float2 v) {
        constexpr int cx = decltype(CX)::value;
        if constexpr (cx == 1) return make_float2(__shfl_up_sync(kFull, v.y, 1), v.x);
        else if constexpr (cx == -1) return make_float2(v.y, __shfl_down_sync(kFull, v.x, 1));
        else return v;
    };
    // slots written now, by 1 + c_z
    int at[3] = {0, 0, 0};
    auto array = [&](int cz, int slot, int index, int count, int base) { return mine + (base + slot * count + index) * kPairArray; };
    float2 before[S::Q];  // populations with c_z = 0 that stay with the thread, made one iteration ago
    static_for_carried<S>([&](auto I) { before[decltype(I)::value] = make_float2(0.f, 0.f); });
    fetch();
    int to = (z0 - 2) * plane + row[1] + col;  // where the next iteration stores, if it does
#pragma unroll 1
    for (int i = 0; i < planes + 2; ++i) {
        float g[S::Q][2], r[S::Q][2];
        static_for_carried<S>([&](auto I) {
            constexpr int v = decltype(I)::value;
            const float2 q = shifted(std::integral_constant<int, S::c(v, 0)>{}, next[v]);
            g[v][0] = q.x;
            g[v][1] = q.y;
        });
        collide_chunk<S>(g, r, cf);
        static_for_carried<S>([&](auto I) {
            constexpr int v = decltype(I)::value, cz = S::c(v, 2);
            if constexpr (pair_shared<S>(v))
                *reinterpret_cast<float2 *>(array(cz, at[1 + cz], pair_count<S>(cz, v), pair_count<S>(cz), pair_base<S>(cz))) =
                    make_float2(r[v][0], r[v][1]);
        });
        __syncthreads();  // the plane's populations are visible; everyone is done with the slots written next
        float2 made[S::Q];
        static_for_carried<S>([&](auto I) {
            constexpr int v = decltype(I)::value;
            if constexpr (!pair_shared<S>(v)) made[v] = make_float2(r[v][0], r[v][1]);
        });
        fetch();  // (the last one of a segment is not used)
        if (i >= 2) {
            static_for_carried<S>([&](auto I) {
                constexpr int v = decltype(I)::value, cy = S::c(v, 1), cz = S::c(v, 2);
                float2 q;
                if constexpr (pair_shared<S>(v)) {
                    constexpr int n = pair_slots(cz), age = 1 + cz;
                    const int slot = at[1 + cz] >= age ? at[1 + cz] - age : at[1 + cz] - age + n;
                    q = *reinterpret_cast<const float2 *>(
                        array(cz, slot, pair_count<S>(cz, v), pair_count<S>(cz), pair_base<S>(cz)) - cy * kPairCols);
                } else {
                    q = cz == -1 ? made[v] : before[v];
                }
                q = shifted(std::integral_constant<int, S::c(v, 0)>{}, q);
                g[v][0] = q.x;
                g[v][1] = q.y;
            });
            collide_chunk<S>(g, r, cf);
            static_for_carried<S>([&](auto I) {
                constexpr int v = decltype(I)::value;
                int o = to;
                asm volatile("" : "+r"(o));
                float *p = dst + v * pitch + o;
                if constexpr (kRagged) {
                    if (live) p[0] = r[v][0];
                    if (live && x + 1 < nx) p[1] = r[v][1];
                } else if (live) {
                    *reinterpret_cast<float2 *>(p) = make_float2(r[v][0], r[v][1]);
                }
            });
        }
        static_for_carried<S>([&](auto I) {
            constexpr int v = decltype(I)::value;
            if constexpr (!pair_shared<S>(v)) before[v] = made[v];
        });
#pragma unroll
        for (int c = 0; c < 3; ++c) at[c] = at[c] + 1 == c + 2 ? 0 : at[c] + 1;
        to += plane;
    }
}

}  // namespace lee
