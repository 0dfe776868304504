// Standalone launch of the fused DUGKS step (tile code in dugks_tile.cuh).
#include <algorithm>

#include "dugks_tile.cuh"
#include "dugks_tile16.cuh"
#include "kin_internal.h"
#include "kin_launch.cuh"
#include "tile_schedule.h"

namespace kin {

// Blocks of TY-row tiles that share an SM.  Two 6-warp blocks (TY <= 5, held to
// 168 registers a thread) run out of step, so one's exchanges overlap the
// other's arithmetic: 0.773 ms at 256^3 against 0.93 for one 9-warp block of
// 8-row tiles and 0.777 for one 12-warp block of 11-row tiles.
constexpr int blocks_per_sm(int ty) { return ty <= 5 ? 2 : 1; }

// Rows that a warp holds whole, where tiles of 30 columns would take two (32^3
// FP32 6.8 -> 5.2 us a step).
constexpr bool whole_rows(int N) { return N == 31 || N == 32; }

// VEL: also write the velocity of the new state to uvel (FP32-computed storage).
template <typename S, int TY, bool VEL, bool WRAP>
__global__ void __launch_bounds__(32 * (TY + 1), sizeof(typename Traits<S>::C) == 4 ? blocks_per_sm(TY) : 1)
    dugks_fused_kernel(const S* __restrict__ src, S* __restrict__ dst, int N, int zchunk,
                       DugksCoef<typename Traits<S>::C> kc, float* __restrict__ uvel) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    grid_begin();
    dugks_tile<S, TY, VEL, WRAP>(src, dst, N, blockIdx.x, blockIdx.y, blockIdx.z, zchunk, kc, smem_raw, uvel);
}

template <typename S, int TY, bool VEL, bool WRAP = false>
static cudaError_t launch_fused_t(const void* src, void* dst, int N, int zchunk,
                                  const DugksCoef<typename Traits<S>::C>& k, float* uvel, cudaStream_t stream) {
    const size_t smem = fused_smem_bytes<S, TY>();
    const cudaError_t e = allow_smem<dugks_fused_kernel<S, TY, VEL, WRAP>>(smem);
    if (e != cudaSuccess) return e;
    if (zchunk <= 0) zchunk = 32;
    if (zchunk > N) zchunk = N;
    dim3 block(32, TY + 1);
    dim3 grid(WRAP ? 1 : (N + 29) / 30, (N + TY - 1) / TY, (N + zchunk - 1) / zchunk);
    return launch_next(dugks_fused_kernel<S, TY, VEL, WRAP>, grid, block, smem, stream, (const S*)src, (S*)dst, N, zchunk, k,
                       uvel);
}

// FP16 and BF16 storage.  EVEN = false: odd N, whose tile reads f-tilde from global
// memory instead of staging it.
template <typename S, int TY, bool VEL, bool EVEN>
__global__ void __launch_bounds__(32 * (TY + 2), 1)
    dugks_fused16_kernel(const S* __restrict__ src, S* __restrict__ dst, int N, int zchunk, DugksCoef<float> kc,
                         float* __restrict__ uvel) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    two_byte::dugks_tile<S, TY, VEL, EVEN>(src, dst, N, blockIdx.x, blockIdx.y, blockIdx.z, zchunk, kc, smem_raw, uvel);
}

template <typename S, int TY, bool VEL, bool EVEN>
static cudaError_t launch_fused16_t(const void* src, void* dst, int N, int zchunk, const DugksCoef<float>& k,
                                    float* uvel, cudaStream_t stream) {
    const size_t smem = two_byte::tile_smem_bytes<S, TY>();
    const cudaError_t e = allow_smem<dugks_fused16_kernel<S, TY, VEL, EVEN>>(smem);
    if (e != cudaSuccess) return e;
    const dim3 grid((N + 29) / 30, (N + TY - 1) / TY, (N + zchunk - 1) / zchunk);
    // an ordinary launch: its copies and, for odd N, its loads go through L1
    dugks_fused16_kernel<S, TY, VEL, EVEN><<<grid, dim3(32, TY + 2), smem, stream>>>((const S*)src, (S*)dst, N, zchunk, k,
                                                                                    uvel);
    return cudaGetLastError();
}

template <typename S, bool VEL>
static cudaError_t launch_fused16(const void* src, void* dst, int N, const DugksCoef<float>& k, int ty, int zchunk,
                                  float* uvel, cudaStream_t stream) {
    if (ty == 4)
        return N % 2 ? launch_fused16_t<S, 4, VEL, false>(src, dst, N, zchunk, k, uvel, stream)
                     : launch_fused16_t<S, 4, VEL, true>(src, dst, N, zchunk, k, uvel, stream);
    return N % 2 ? launch_fused16_t<S, 8, VEL, false>(src, dst, N, zchunk, k, uvel, stream)
                 : launch_fused16_t<S, 8, VEL, true>(src, dst, N, zchunk, k, uvel, stream);
}

template <typename S, bool VEL>
static cudaError_t launch_fused_v(const void* src, void* dst, int N, const DugksCoef<typename Traits<S>::C>& k,
                                  int ty, int zchunk, float* uvel, cudaStream_t stream) {
    if constexpr (sizeof(typename Traits<S>::C) == 8) {
        if (ty == 3 && whole_rows(N)) return launch_fused_t<S, 3, VEL, true>(src, dst, N, zchunk, k, uvel, stream);
        if (ty == 3) return launch_fused_t<S, 3, VEL>(src, dst, N, zchunk, k, uvel, stream);
        return launch_fused_t<S, 7, VEL>(src, dst, N, zchunk, k, uvel, stream);
    } else if constexpr (sizeof(S) == 2) {
        return launch_fused16<S, VEL>(src, dst, N, k, ty, zchunk, uvel, stream);
    } else {
        if (ty == 8 && whole_rows(N)) return launch_fused_t<S, 8, VEL, true>(src, dst, N, zchunk, k, uvel, stream);
        switch (ty) {
            case 4: return launch_fused_t<S, 4, VEL>(src, dst, N, zchunk, k, uvel, stream);
            case 5: return launch_fused_t<S, 5, VEL>(src, dst, N, zchunk, k, uvel, stream);
            case 8: return launch_fused_t<S, 8, VEL>(src, dst, N, zchunk, k, uvel, stream);
            case 11: return launch_fused_t<S, 11, VEL>(src, dst, N, zchunk, k, uvel, stream);
        }
        return cudaErrorInvalidValue;
    }
}

template <typename S>
static cudaError_t launch_fused(const void* src, void* dst, int N, double nu, double dt, int ty,
                                int zchunk, float* uvel, cudaStream_t stream) {
    using C = typename Traits<S>::C;
    const DugksCoef<C> k = dugks_coef<C>(nu, dt);
    if constexpr (sizeof(C) == 8) {
        if (uvel) return cudaErrorInvalidValue;  // FP64 storage keeps the FP64 statistics path
    } else {
        if (uvel) return launch_fused_v<S, true>(src, dst, N, k, ty, zchunk, uvel, stream);
    }
    return launch_fused_v<S, false>(src, dst, N, k, ty, zchunk, nullptr, stream);
}

KIN_DEBUG_ACCESSOR(debug_word_dugks)

cudaError_t dugks_step_fused(int storage, const void* src, void* dst, int N, double nu, double dt,
                             int ty, int zchunk, cudaStream_t stream, float* uvel) {
    switch (storage) {
        case ST_F32: return launch_fused<float>(src, dst, N, nu, dt, ty, zchunk, uvel, stream);
        case ST_F16: return launch_fused<__half>(src, dst, N, nu, dt, ty, zchunk, uvel, stream);
        case ST_BF16: return launch_fused<__nv_bfloat16>(src, dst, N, nu, dt, ty, zchunk, uvel, stream);
        case ST_F64: return launch_fused<double>(src, dst, N, nu, dt, ty, zchunk, uvel, stream);
    }
    return cudaErrorInvalidValue;
}

namespace {

// What the launch shape is chosen among, with the measured time of one plane
// of a block (us): alone on its SM and with the SM's blocks all there.  FP64: a
// row costs about 18 us of one scheduler's FP64 pipe a plane, so blocks are 4 or 8
// warps, one or two a scheduler: five (4-row tiles) took as long as eight
// (32^3 148 -> 90 us a step, 128^3 4.24 -> 3.55 ms).
struct TileShape {
    int ty, per_sm;
    double alone, shared;
    bool wraps;  // has the whole-row form
};
constexpr TileShape kShapes[] = {{4, 2, 1.5, 1.85, false}, {5, 2, 1.28, 2.0, false}, {8, 1, 1.76, 1.76, true}, {11, 1, 2.1, 2.1, false}};
constexpr TileShape kShapes64[] = {{3, 1, 21.3, 21.3, true}, {7, 1, 41.5, 41.5, false}};

constexpr long long kMaxBlocks = 20000;  // of a grid that is considered

long long columns(int N, const TileShape& t) {
    const int ty = t.ty;
    const bool wrap = whole_rows(N) && t.wraps;
    return (long long)(wrap ? 1 : (N + 29) / 30) * ((N + ty - 1) / ty);
}

// Time (us) of the fused DUGKS launch with tiles of shape t and z chunks of zc
// planes; a block's prologue (two pre-steps and one record before the first
// face) takes about 1.1 plane-times.
double makespan(int N, const TileShape& t, int zc, int nsm) {
    const long long cols = columns(N, t);
    const double plane = cols * ((N + zc - 1) / zc) <= nsm ? t.alone : t.shared;
    return plane * tile_schedule(cols, N, zc, (long long)nsm * t.per_sm, 1.1);
}

// Planes per block of the FP16 and BF16 step, one block an SM with a prologue of 1.5
// plane-times: from 1.5 waves of columns on chunks that make about two waves of
// blocks (256^3: 240 + 16 planes, the measured optimum), else the length with the
// shortest schedule.  Lengths that leave a shorter last chunk are tried too: its
// blocks fill the last wave (us a step against even chunks: 88^3 47.3 / 51.4, 128^3
// 155 / 165, 192^3 439 / 455).
int two_byte_zchunk(int N, int ty, int nsm) {
    const long long cols = (long long)((N + 29) / 30) * ((N + ty - 1) / ty);
    if (2 * cols >= 3LL * nsm)
        return (int)std::max(8LL, std::min<long long>((long long)N * cols / (2LL * nsm) / 8 * 8, N));
    double best = -1.0;
    int zc = N;
    for (int c = N; c >= 1; --c) {
        const int nz = (N + c - 1) / c;
        if (nz > 1 && (nz > 64 || cols * nz > kMaxBlocks)) break;
        const double m = tile_schedule(cols, N, c, nsm, 1.5);
        if (best < 0.0 || m < best * (1.0 - 0.005)) {
            best = m;
            zc = c;
        }
    }
    return zc;
}

}  // namespace

// The step lasts as long as its busiest SM, so a chunk length that leaves the
// last wave nearly empty costs up to a third of it.  Every tile height and
// chunk length is scored by the schedule above and the shortest taken (the
// longest chunk among those within 0.5 %: fewer halo planes).  Measured against
// sweeps of all shapes (before steps overlapped the end of the step before,
// which took ~2 us off the small ones): 33^3 8 x 2 planes 7.6 us, 48^3 8 x 4 12.3
// us (5 x 8: 14.4), 64^3 11 x 8 22.5 us (8 x 11: 23.8), 97^3 11 x 25 61.6 us
// (5 x 13: 66.6), 128^3 11 x 26 117 us (5 x 19: 119), 256^3 11 x 37 0.777 ms
// (5 x 52: 0.773).
void dugks_fused_shape(int storage, int N, int nsm, int want_ty, int want_zc, int* ty, int* zc) {
    double best = -1.0;
    auto consider = [&](const TileShape& t) {
        const long long cols = columns(N, t);
        for (int c = want_zc > 0 ? std::min(want_zc, N) : N; c >= 1; --c) {
            const int nz = (N + c - 1) / c;
            if (want_zc <= 0 && nz > 1 && (nz > 64 || cols * nz > kMaxBlocks)) break;
            // of the lengths that give nz chunks, the smallest is the most even
            if (want_zc <= 0 && c > 1 && (N + c - 2) / (c - 1) == nz) continue;
            const double m = makespan(N, t, c, nsm);
            if (best < 0.0 || m < best * (1.0 - 0.005)) {
                best = m;
                *ty = t.ty;
                *zc = c;
            }
            if (want_zc > 0) break;
        }
    };
    if (storage == ST_F64) {
        for (const TileShape& t : kShapes64) consider(t);
        return;
    }
    if (storage != ST_F32) {
        *ty = want_ty == 4 ? 4 : 8;
        *zc = want_zc > 0 ? std::min(want_zc, N) : two_byte_zchunk(N, *ty, nsm);
        return;
    }
    for (const TileShape& t : kShapes)
        if (want_ty > 0 ? t.ty == want_ty : t.ty != 4) consider(t);
}

}  // namespace kin
