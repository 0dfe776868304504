// Standalone launch of the MRT-LBE step (node update in lbe_node.cuh).
// HBM traffic per node: 19 loads + 19 stores of the storage type.
#include "kin_internal.h"
#include "kin_launch.cuh"
#include "lbe_node.cuh"
#include "lbe_pair.cuh"
#include "tile_schedule.h"

#include <algorithm>
#include <cstring>

namespace kin {

// Blocks of b threads along x.  In boxes of up to 64 two rows of 33..64 threads
// share a block (64^3 FP32 5.2 us a step instead of 6.2, 48^3 3.8 instead of
// 3.9); one-warp rows stay apart (32^3 3.5 us against 4.0 with four rows a
// block), and in larger boxes a row fills a block or the rows are many
// (256^3 FP16: 214 us either way).  Where 32 threads are asked for in a longer row,
// warps is the rows that share a block (one cell a thread, FP32: 4; blocks of one warp
// each pay the overlapped start, 256^3 529 us, 372 with four rows).
static void step_shape(int nx, int N, int b, int warps, dim3& block, dim3& grid) {
    const int bx = std::min(b, ((nx + 31) / 32) * 32);
    const int by = bx >= 64 && N <= 64 ? std::max(1, b / bx) : bx == 32 && nx > 32 ? warps : 1;
    block = dim3(bx, by);
    grid = dim3((nx + bx - 1) / bx, (N + by - 1) / by, N);
}

template <typename S>
__global__ void __launch_bounds__(256) lbe_step_kernel(const S* __restrict__ src,
                                                       S* __restrict__ dst, int N, size_t plane,
                                                       MrtRates<typename Traits<S>::C> rates) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    grid_begin();
    if (x >= N || y >= N) return;
    lbe_node<S>(src, dst, N, plane, x, y, blockIdx.z, rates);
}

template <typename S, int V>
__global__ void __launch_bounds__(256) lbe_stepv_kernel(const S* __restrict__ src, S* __restrict__ dst,
                                                        int N, size_t plane, MrtRates<float> rates) {
    const int x = V * (blockIdx.x * blockDim.x + threadIdx.x);
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    grid_begin();
    if (x >= N || y >= N) return;
    lbe_vnode<S, V>(src, dst, N, plane, x, y, blockIdx.z, rates);
}

// Four cells a thread with the populations held packed (lbe_vnode4p), held to
// 96 registers instead of the 128 that four cells' 76 floats take, so that
// more warps are resident: 0.222 -> 0.214 ms (FP16) at 256^3, bitwise the
// same results.
template <typename S>
__global__ void __maxnreg__(96) lbe_stepv4_kernel(const S* __restrict__ src, S* __restrict__ dst, int N,
                                                  size_t plane, MrtRates<float> rates) {
    const int x = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    grid_begin();
    if (x >= N || y >= N) return;
    lbe_vnode4p<S>(src, dst, N, plane, x, y, blockIdx.z, rates);
}

template <typename S, int V>
static cudaError_t launch_lbe_v(const S* src, S* dst, int N, const MrtRates<float>& r, int bx,
                                cudaStream_t stream) {
    const int nv = N / V;
    int b = bx > 0 ? std::min(bx, 256) : 128;
    dim3 block, grid;
    step_shape(nv, N, b, 1, block, grid);
    const size_t plane = (size_t)N * N * N;
    if constexpr (V == 4) return launch_next(lbe_stepv4_kernel<S>, grid, block, 0, stream, src, dst, N, plane, r);
    else return launch_next(lbe_stepv_kernel<S, V>, grid, block, 0, stream, src, dst, N, plane, r);
}

// An FP64 step of a few warps an SM is bound by the busiest scheduler's FP64 pipe.
// Blocks that wait beside the grid before them are placed around its warps, so that
// some schedulers get several and others none; the ordinary launch spreads them
// evenly.  us a step overlapped / ordinary: 16^3 6.7 / 8.2, 19^3 6.8 / 9.1, 20^3 28.8 /
// 8.2, 24^3 29.2 / 10.3, 32^3 30.2 / 14.4, 34^3 31.1 / 26.8, 35^3 31.2 / 32.8, 48^3
// 48.6 / 51.2, 64^3 84.0 / 86.1 (361 warps at 19^3, 400 at 20^3, 2312 at 34^3, 2520 at
// 35^3; 2.5 and 16 warps an SM are 380 and 2432).
static bool overlap_unbalances(const dim3& grid, const dim3& block, int nsm) {
    const long long warps = (long long)grid.x * grid.y * grid.z * (block.x * block.y / 32);
    return 2 * warps > 5LL * nsm && warps < 16LL * nsm;
}

template <typename S>
static cudaError_t launch_lbe(const void* src, void* dst, int N, double nu, int bx, int nsm,
                              cudaStream_t stream) {
    using C = typename Traits<S>::C;
    const MrtRates<C> r = lbe_rates<C>(nu);
    if constexpr (sizeof(S) == 2) {
        if (N % 4 == 0) return launch_lbe_v<S, 4>((const S*)src, (S*)dst, N, r, bx, stream);
        if (N % 2 == 0) return launch_lbe_v<S, 2>((const S*)src, (S*)dst, N, r, bx, stream);
    }
    if (bx <= 0) bx = 128;
    if (bx > 256) bx = 256;  // the kernel's launch bounds
    dim3 block, grid;
    step_shape(N, N, bx, sizeof(C) == 8 ? 1 : 4, block, grid);
    if (sizeof(C) == 8 && overlap_unbalances(grid, block, nsm)) {
        lbe_step_kernel<S><<<grid, block, 0, stream>>>((const S*)src, (S*)dst, N, (size_t)N * N * N, r);
        return cudaGetLastError();
    }
    return launch_next(lbe_step_kernel<S>, grid, block, 0, stream, (const S*)src, (S*)dst, N, (size_t)N * N * N, r);
}

// One iteration of the consistent initialisation (Sec. IV.A, after Mei et
// al.): the node update of lbe_node with the momentum held at rho0 u0 (FP64,
// [3][N^3]); see mrt_collide_t.
template <typename S>
__global__ void __launch_bounds__(256) lbe_consistent_kernel(const S* __restrict__ src, S* __restrict__ dst,
                                                             int N, size_t plane,
                                                             MrtRates<typename Traits<S>::C> rates,
                                                             const double* __restrict__ u0) {
    using C = typename Traits<S>::C;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= N) return;
    const int y = blockIdx.y, z = blockIdx.z;
    C f[Q];
    lbe_gather<S>(src, N, plane, x, y, z, f);
    const size_t c = (size_t)x + (size_t)N * (y + (size_t)N * z);
    mrt_collide_as<S, true>(f, rates, (C)u0[c], (C)u0[plane + c], (C)u0[2 * plane + c]);
    lbe_scatter<S>(dst, N, plane, x, y, z, f);
}

template <typename S>
static cudaError_t launch_consistent(const void* src, void* dst, int N, double nu, const double* u0,
                                     cudaStream_t stream) {
    using C = typename Traits<S>::C;
    const int bx = N >= 128 ? 128 : ((N + 31) / 32) * 32;
    dim3 block(bx), grid((N + bx - 1) / bx, N, N);
    lbe_consistent_kernel<S><<<grid, block, 0, stream>>>((const S*)src, (S*)dst, N, (size_t)N * N * N,
                                                         lbe_rates<C>(nu), u0);
    return cudaGetLastError();
}

cudaError_t lbe_consistent_step(int storage, const void* src, void* dst, int N, double nu, const double* u0,
                                cudaStream_t stream) {
    switch (storage) {
        case ST_F32: return launch_consistent<float>(src, dst, N, nu, u0, stream);
        case ST_F16: return launch_consistent<__half>(src, dst, N, nu, u0, stream);
        case ST_BF16: return launch_consistent<__nv_bfloat16>(src, dst, N, nu, u0, stream);
        case ST_F64: return launch_consistent<double>(src, dst, N, nu, u0, stream);
    }
    return cudaErrorInvalidValue;
}

// Two steps in one launch pay where a step is mostly the hand-over between two
// grids (us a step, single / paired, FP32: 8^3 1.6 / 1.3, 24^3 2.0 / 1.35, 32^3
// 3.5 / 1.4), and where the state does not stay in L2 between steps (64^3 5.2 /
// 7.6, 40 MB of state; 84^3 11.8 / 12.1, 88^3 14.1 / 12.2, 97^3 24.6 / 21.0, 128^3
// 47.9 / 37.9, 256^3 367 / 257).  2-byte steps of large boxes are bound by their
// operations, FP64 always is.
bool lbe_pairs(int storage, int N) { return N <= 32 ? storage != ST_F64 : storage == ST_F32 && N >= 88; }

template <typename S>
static cudaError_t launch_small_pair(const void* src, void* dst, int N, double nu, cudaStream_t stream) {
    // 96 blocks of 768 threads at 32^3; 6 rows x 1 plane 2.4 us a step, 6 x 2 1.6,
    // 3 x 2 2.1, 8 x 1 1.5, 2 x 2 1.75
    constexpr int TY = 4, TZ = 2;
    constexpr size_t smem = sizeof(float) * Q * 32 * (TY + 2) * (TZ + 2);
    cudaError_t e = allow_smem<lbe_small_pair_kernel<S, TY, TZ>>(smem);
    if (e != cudaSuccess) return e;
    return launch_next(lbe_small_pair_kernel<S, TY, TZ>, dim3((N + TY - 1) / TY, (N + TZ - 1) / TZ),
                       dim3(32, TY + 2, TZ + 2), smem, stream, (const S*)src, (S*)dst, N, (size_t)N * N * N,
                       lbe_rates<float>(nu));
}

cudaError_t lbe_pair_step(int storage, const void* src, void* dst, int N, double nu, int nsm, cudaStream_t stream) {
    if (!lbe_pairs(storage, N)) return cudaErrorInvalidValue;
    if (N <= 32) {
        if (storage == ST_F32) return launch_small_pair<float>(src, dst, N, nu, stream);
        if (storage == ST_F16) return launch_small_pair<__half>(src, dst, N, nu, stream);
        return launch_small_pair<__nv_bfloat16>(src, dst, N, nu, stream);
    }
    constexpr int TY = kPairRows;
    constexpr size_t smem = sizeof(float) * LbePairSmem<TY>::FLOATS;
    cudaError_t e = allow_smem<lbe_pair_kernel<TY>>(smem);
    if (e != cudaSuccess) return e;
    // planes a block: the shortest schedule, of at most 64 chunks (a block relaxes
    // two planes before its first result)
    const long long cols = (long long)((N + 29) / 30) * ((N + TY - 1) / TY);
    int zc = N;
    double best = -1.0;
    for (int nz = 1; nz <= 64 && nz <= N; ++nz) {
        const int c = (N + nz - 1) / nz;
        const double t = tile_schedule(cols, N, c, (long long)nsm * kPairBlocks, 2.0);
        if (best < 0.0 || t < best) {
            best = t;
            zc = c;
        }
    }
    const dim3 grid((N + 29) / 30, (N + TY - 1) / TY, (N + zc - 1) / zc);
    return launch_next(lbe_pair_kernel<TY>, grid, dim3(32, TY + 2), smem, stream, (const float*)src, (float*)dst, N,
                       (size_t)N * N * N, zc, lbe_rates<float>(nu));
}

KIN_DEBUG_ACCESSOR(debug_word_lbe)

cudaError_t lbe_step(int storage, const void* src, void* dst, int N, double nu, int block_x, int nsm,
                     cudaStream_t stream) {
    switch (storage) {
        case ST_F32: return launch_lbe<float>(src, dst, N, nu, block_x, nsm, stream);
        case ST_F16: return launch_lbe<__half>(src, dst, N, nu, block_x, nsm, stream);
        case ST_BF16: return launch_lbe<__nv_bfloat16>(src, dst, N, nu, block_x, nsm, stream);
        case ST_F64: return launch_lbe<double>(src, dst, N, nu, block_x, nsm, stream);
    }
    return cudaErrorInvalidValue;
}

}  // namespace kin
