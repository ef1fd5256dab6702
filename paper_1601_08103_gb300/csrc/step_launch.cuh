// step_launch.cuh -- launch configuration of the fused stream-collide kernels for one velocity set:
// the one-step kernel (cells per thread, grid), the 2D row pipeline (segment height from the
// resident capacity) and the 3D plane pipelines (tiles and segments likewise).  Together with
// kernels.cuh, rowpipe.cuh and velsets.cuh this fixes what the profiled hot-path launches execute.
#pragma once

#include "ops.cuh"
#include "planepair.cuh"
#include "planepipe.cuh"
#include "rowpipe.cuh"

namespace lee {

template <class S, class T, int V, Edge EDGE, bool CUT = false>
cudaError_t launch_step_v(const StepLaunch &L) {
    using C = typename Store<T>::C;
    GridDesc gd;
    gd.nx = L.nx;
    gd.ny = L.ny;
    gd.nz = L.nz;
    gd.nxc = L.nx / V;
    gd.nchunks = (long long)gd.nxc * L.ny * L.nz;
    gd.pitch = L.pitch;
    const CollideCoef<C> cf = make_coef<C>(L.omega, L.coefM, L.coefN);
    OpenEdge<C> ob;
    ob.sponge_w = L.sponge_w;
    ob.sponge_smax = (C)L.sponge_smax;
    ob.ghost = static_cast<const C *>(L.ghost);
    ob.ghost_L = L.ghost_L;
    ob.skip_border = L.skip_border;
    const long long blocks = (gd.nchunks + 255) / 256;
    k_stream_collide<S, T, V, EDGE, CUT><<<(unsigned)blocks, 256, 0, L.stream>>>(static_cast<const T *>(L.src),
                                                                                   static_cast<T *>(L.dst), gd, cf, ob);
    return cudaGetLastError();
}

template <class S, class T, int V>
cudaError_t launch_step_edge(const StepLaunch &L) {
    if (!L.open) return launch_step_v<S, T, V, kWrapEdge>(L);
    if constexpr (S::D == 2) {
        if (L.ghost || L.skip_border) return launch_step_v<S, T, V, kGhostEdge>(L);
    }
    if (L.ghost || L.skip_border) return cudaErrorInvalidValue;
    // (D3Q19: its zero edge runs 5 % slower in an instance of its own, 192^3 FP32 209 against 198 us per step)
    if constexpr (rest_static<S>()) {
        if (L.sponge_w == 0) return launch_step_v<S, T, V, kZeroEdge>(L);
    }
    return launch_step_v<S, T, V, kFrameEdge>(L);
}

// Vector width: one 16-byte access per velocity and thread (8 bytes for the 19-velocity set, to
// bound register use); one cell per thread when nx is not a multiple of the width.
template <class S, class T>
constexpr int vec_width() {
    constexpr int bytes = (S::Q > 13) ? 8 : 16;
    constexpr int v = bytes / (int)sizeof(T);
    return v < 1 ? 1 : v;
}

// BFP16 storage (bfp.cuh): 8 cells per lane (4 for the 13- and 19-velocity sets, which would
// need 128 registers at 8; LEE_BFP_CELLS=4 or 8 at create time picks either, for comparisons)
// when nx is a multiple of the 8-cell block, one cell per lane otherwise.
template <class S, int V, Edge EDGE>
cudaError_t launch_step_bfp_v(const StepLaunch &L) {
    GridDesc gd;
    gd.nx = L.nx;
    gd.ny = L.ny;
    gd.nz = L.nz;
    gd.nxc = L.nx / V;
    gd.nchunks = (long long)gd.nxc * L.ny * L.nz;
    gd.pitch = L.pitch;
    const CollideCoef<float> cf = make_coef<float>(L.omega, L.coefM, L.coefN);
    const OpenEdge<float> ob{L.sponge_w, (float)L.sponge_smax, nullptr, 0};
    const long long blocks = (gd.nchunks + 255) / 256;
    k_stream_collide_bfp<S, V, EDGE><<<(unsigned)blocks, 256, 0, L.stream>>>(static_cast<const Bfp16 *>(L.src),
                                                                               static_cast<Bfp16 *>(L.dst), gd, cf, ob);
    return cudaGetLastError();
}
template <class S, int V>
cudaError_t launch_step_bfp_edge(const StepLaunch &L) {
    return !L.open ? launch_step_bfp_v<S, V, kWrapEdge>(L)
           : L.sponge_w > 0 ? launch_step_bfp_v<S, V, kFrameEdge>(L) : launch_step_bfp_v<S, V, kZeroEdge>(L);
}
template <class S>
cudaError_t launch_step_bfp(const StepLaunch &L) {
    if (L.ghost) return cudaErrorInvalidValue;  // no learned edge on BFP16 storage
    if (!L.force_scalar && L.nx % kBfpBlock == 0) {
        const int V = L.bfp_cells ? L.bfp_cells : (S::Q > 9 ? 4 : 8);
        return V == 4 ? launch_step_bfp_edge<S, 4>(L) : launch_step_bfp_edge<S, 8>(L);
    }
    return launch_step_bfp_edge<S, 1>(L);
}

template <class S, class T>
cudaError_t launch_step_t(const StepLaunch &L) {
    if constexpr (std::is_same<T, Bfp16>::value) {
        return launch_step_bfp<S>(L);
    } else {
        constexpr int V = vec_width<S, T>();
        if constexpr (S::D >= 2) {
            if (L.slab) {  // periodic except along the cut, which reads the halo planes
                if constexpr (V > 1) {
                    if (!L.force_scalar && L.nx % V == 0) return launch_step_v<S, T, V, kWrapEdge, true>(L);
                }
                return launch_step_v<S, T, 1, kWrapEdge, true>(L);
            }
        }
        if constexpr (V > 1) {
            if (!L.force_scalar && L.nx % V == 0) return launch_step_edge<S, T, V>(L);
        }
        return launch_step_edge<S, T, 1>(L);
    }
}

template <class Fn>
cudaError_t with_storage(int storage, Fn &&fn) {
    switch (storage) {
    case LEE_STORE_F64: return fn((double *)nullptr);
    case LEE_STORE_F32: return fn((float *)nullptr);
    case LEE_STORE_F16: return fn((__half *)nullptr);
    case LEE_STORE_BF16: return fn((__nv_bfloat16 *)nullptr);
    case LEE_STORE_BFP16: return fn((Bfp16 *)nullptr);
    default: return cudaErrorInvalidValue;
    }
}

// Row pipeline (rowpipe.cuh): the resident warps of a device, set by row_pipe_prepare outside any
// stream capture, and the launch.
template <int K, class IO, int kStages>
int *row_pipe_capacity() {
    static int cap[64] = {0};
    return cap;
}
template <int K, class IO, int kStages>
cudaError_t row_pipe_prepare_stages() {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (row_pipe_capacity<K, IO, kStages>()[dev]) return cudaSuccess;
    constexpr int smem = rp_smem_bytes<IO, kStages>();
    int per_sm = 0, sms = 0;
    e = cudaFuncSetAttribute(k_row_pipe<K, IO, kStages>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_row_pipe<K, IO, kStages>, 32 * kRpWarps, smem);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    row_pipe_capacity<K, IO, kStages>()[dev] = per_sm * sms > 0 ? per_sm * sms * kRpWarps : 1;
    return cudaSuccess;
}
template <int K, class IO, int kStages>
cudaError_t row_pipe_launch_stages(const StepLaunch &L) {
    using E = typename IO::Elem;
    if (L.open || (!IO::kRagged && L.nx % IO::kAlign != 0)) return cudaErrorInvalidValue;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    const int capacity = row_pipe_capacity<K, IO, kStages>()[dev];
    if (capacity == 0) return cudaErrorNotReady;  // prepare first
    const CollideCoef<float> cf = make_coef<float>(L.omega, L.coefM, L.coefN);
    // segment height: the smallest even number (at least kRpMinRows) that puts every tile in one resident
    // wave (twice or half as many warps measured 10 to 40 % slower on 2048^2 .. 8192^2)
    constexpr int width = rp_width<K, IO>();
    const int strips = (L.nx + width - 1) / width;
    const int segs = capacity / strips > 1 ? capacity / strips : 1;
    int H = (L.ny + segs - 1) / segs;
    H += H & 1;
    if (H < kRpMinRows) H = kRpMinRows;
    const int tiles = strips * ((L.ny + H - 1) / H);
    k_row_pipe<K, IO, kStages><<<(tiles + kRpWarps - 1) / kRpWarps, 32 * kRpWarps, rp_smem_bytes<IO, kStages>(),
                                 L.stream>>>(static_cast<const E *>(L.src), static_cast<E *>(L.dst), L.nx, L.ny, L.pitch,
                                             H, strips, tiles, cf.M[1][1]);
    return cudaGetLastError();
}
template <int K, class IO>
cudaError_t row_pipe_prepare() {
    if constexpr (std::is_base_of<RpF32, IO>::value) {
        const cudaError_t e = row_pipe_prepare_stages<K, IO, kRpStagesNear>();
        return e != cudaSuccess ? e : row_pipe_prepare_stages<K, IO, kRpStagesFar>();
    } else {
        return row_pipe_prepare_stages<K, IO, kRpStages16>();
    }
}
template <int K, class IO>
cudaError_t row_pipe_launch(const StepLaunch &L) {
    if constexpr (std::is_base_of<RpF32, IO>::value) {
        return 8LL * (long long)sizeof(float) * L.nx * L.ny <= kRpNearL2Bytes
                   ? row_pipe_launch_stages<K, IO, kRpStagesNear>(L)
                   : row_pipe_launch_stages<K, IO, kRpStagesFar>(L);
    } else {
        return row_pipe_launch_stages<K, IO, kRpStages16>(L);
    }
}

// Plane pipeline (planepipe.cuh): its cut of a grid, made once by plane_pipe_prepare (the search takes tens of
// microseconds), and the launch.
template <bool kRagged>
int *plane_pipe_capacity() {
    static int cap[64] = {0};
    return cap;
}
// The resident blocks of `kern` on the current device, kept in cap[device] and asked for outside any stream
// capture.
template <class Kern>
cudaError_t resident_blocks(Kern kern, int threads, int smem, int *cap, int &blocks) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (cap[dev] == 0) {
        int per_sm = 0, sms = 0;
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        cap[dev] = per_sm * sms > 0 ? per_sm * sms : 1;
    }
    blocks = cap[dev];
    return cudaSuccess;
}
template <bool kRagged>
cudaError_t plane_pipe_prepare_for(int nx, int ny, int nz, int (&cut)[4]) {
    int blocks = 0;
    const cudaError_t e = resident_blocks(k_plane_pipe<kPpDeep, kRagged>, kPpThreads, pp_smem_bytes<kPpDeep>(),
                                          plane_pipe_capacity<kRagged>(), blocks);
    if (e != cudaSuccess) return e;
    const PpCut c = plane_pipe_cut(kPpDeep, pp_halo<kPpDeep>(), nx, ny, nz, blocks);
    cut[0] = c.C;
    cut[1] = c.width;
    cut[2] = c.height;
    cut[3] = c.HZ;
    return cudaSuccess;
}
template <bool kRagged>
cudaError_t plane_pipe_launch_for(const StepLaunch &L) {
    const PpCut cut{L.cut3d[0], L.cut3d[1], L.cut3d[2], L.cut3d[3]};
    const long long gy = cut.C ? (L.ny + cut.height - 1) / cut.height : 0, gz = cut.C ? (L.nz + cut.HZ - 1) / cut.HZ : 0;
    if (cut.C == 0 || gy > 65535 || gz > 65535) return cudaErrorInvalidValue;
    const CollideCoef<float> cf = make_coef<float>(L.omega, L.coefM, L.coefN);
    k_plane_pipe<kPpDeep, kRagged><<<dim3((L.nx + cut.width - 1) / cut.width, (unsigned)gy, (unsigned)gz), kPpThreads,
                                     pp_smem_bytes<kPpDeep>(), L.stream>>>(
        static_cast<const float *>(L.src), static_cast<float *>(L.dst), L.nx, L.ny, L.nz, L.pitch, cut, cf.M[1][1]);
    return cudaGetLastError();
}
inline cudaError_t plane_pipe_prepare(int nx, int ny, int nz, int (&cut)[4]) {
    return nx % 4 == 0 ? plane_pipe_prepare_for<false>(nx, ny, nz, cut) : plane_pipe_prepare_for<true>(nx, ny, nz, cut);
}
inline cudaError_t plane_pipe_launch(const StepLaunch &L) {
    if (L.storage != LEE_STORE_F32 || L.open) return cudaErrorInvalidValue;
    return L.nx % 4 == 0 ? plane_pipe_launch_for<false>(L) : plane_pipe_launch_for<true>(L);
}

// Two steps per launch of the sets with diagonal velocities (planepair.cuh), likewise.
template <class S, bool kRagged>
int *plane_pair_capacity() {
    static int cap[64] = {0};
    return cap;
}
template <class S, bool kRagged>
cudaError_t plane_pair_prepare_for(int nx, int ny, int nz, int (&cut)[4]) {
    int blocks = 0;
    const cudaError_t e = resident_blocks(k_plane_pair<S, kRagged>, kPairThreads, pair_smem_bytes<S>(),
                                          plane_pair_capacity<S, kRagged>(), blocks);
    if (e == cudaSuccess) cut[3] = plane_pair_segment(nx, ny, nz, blocks);
    return e;
}
template <class S, bool kRagged>
cudaError_t plane_pair_launch_for(const StepLaunch &L) {
    const int HZ = L.cut3d[3];
    const long long gy = (L.ny + kPairHeight - 1) / kPairHeight;
    if (HZ == 0 || gy > 65535) return cudaErrorInvalidValue;
    k_plane_pair<S, kRagged><<<dim3((L.nx + kPairWidth - 1) / kPairWidth, (unsigned)gy, (L.nz + HZ - 1) / HZ),
                               kPairThreads, pair_smem_bytes<S>(), L.stream>>>(
        static_cast<const float *>(L.src), static_cast<float *>(L.dst), L.nx, L.ny, L.nz, L.pitch, HZ,
        make_coef<float>(L.omega, L.coefM, L.coefN));
    return cudaGetLastError();
}
template <class S>
cudaError_t plane_pair_prepare(int nx, int ny, int nz, int (&cut)[4]) {
    return nx % 2 == 0 ? plane_pair_prepare_for<S, false>(nx, ny, nz, cut) : plane_pair_prepare_for<S, true>(nx, ny, nz, cut);
}
template <class S>
cudaError_t plane_pair_launch(const StepLaunch &L) {
    if (L.storage != LEE_STORE_F32 || L.open) return cudaErrorInvalidValue;
    return L.nx % 2 == 0 ? plane_pair_launch_for<S, false>(L) : plane_pair_launch_for<S, true>(L);
}

}  // namespace lee
