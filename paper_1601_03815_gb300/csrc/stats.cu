// Statistics and state conversion kernels.
//
//   velocity_kernel        u = sum xi_i f_i (Eq. 8 / Eq. 12), FP64 out
//   velocity32_kernel      the same in FP32, for storage types computed in FP32
//   ed_partial_kernel      per-block FP64 sums of |u|^2 and s_ab s_ab
//   ed32_partial_kernel    the same from FP32 u: per-cell terms in FP32,
//                          per-thread and block sums in FP64
//                          (the last block of either to finish sums the
//                          partials in a fixed order -> {E, eps})
//   ed_final_kernel        that sum as a kernel, for callers without the
//                          counter that tells the last block
//   shell_partial_kernel   per-block shell sums of |u_hat|^2 / 2 (Eq. 27)
//   shell_final_kernel     fixed-order sum over blocks
// Every reduction runs in a fixed order for a given N, so results are
// bitwise reproducible.
#include "kin.h"
#include "kin_common.cuh"
#include "kin_internal.h"
#include "kin_launch.cuh"
#include "kin_sim.h"
#include "lbe_node.cuh"

#include <cufft.h>

#include <algorithm>

namespace kin {

size_t storage_bytes(int storage) {
    switch (storage) {
        case ST_F32: return 4;
        case ST_F16: return 2;
        case ST_BF16: return 2;
        case ST_F64: return 8;
    }
    return 0;
}

// Canonical cell index of the stored element of population I for node x: the
// LBE pull layout stores f_i(x) at x - xi_i.
template <int I>
__device__ __forceinline__ int stored_index(int x, int y, int z, int N, bool shifted) {
    if (!shifted) return x + N * (y + N * z);
    int xs = x - cx(I), ys = y - cy(I), zs = z - cz(I);
    xs = xs < 0 ? xs + N : (xs >= N ? xs - N : xs);
    ys = ys < 0 ? ys + N : (ys >= N ? ys - N : ys);
    zs = zs < 0 ? zs + N : (zs >= N ? zs - N : zs);
    return xs + N * (ys + N * zs);
}

__device__ __forceinline__ int stored_index_rt(int i, int x, int y, int z, int N, bool shifted) {
    if (!shifted) return x + N * (y + N * z);
    int xs = x - cx(i), ys = y - cy(i), zs = z - cz(i);
    xs = xs < 0 ? xs + N : (xs >= N ? xs - N : xs);
    ys = ys < 0 ? ys + N : (ys >= N ? ys - N : ys);
    zs = zs < 0 ? zs + N : (zs >= N ? zs - N : zs);
    return xs + N * (ys + N * zs);
}

template <typename S>
__global__ void velocity_kernel(const S* __restrict__ st, bool shifted, int N, size_t plane,
                                double* __restrict__ u) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    grid_begin();
    if (x >= N) return;
    const int y = blockIdx.y, z = blockIdx.z;
    // 21 FP64 additions: an opposite pair enters as its difference
    double b[NPAIR];
    static_for<0, NPAIR>([&](auto pc) {
        constexpr int P = decltype(pc)::value, I = 2 * P + 1;
        b[P] = (double)Traits<S>::load_l2(st + I * plane + stored_index<I>(x, y, z, N, shifted)) -
               (double)Traits<S>::load_l2(st + (I + 1) * plane + stored_index<I + 1>(x, y, z, N, shifted));
    });
    const double jx = (b[0] + b[3]) + (b[4] + (b[5] + b[6]));
    const double jy = (b[1] + b[3]) - (b[4] - (b[7] + b[8]));
    const double jz = (b[2] + b[5]) - (b[6] - (b[7] - b[8]));
    const size_t c = (size_t)x + (size_t)N * (y + (size_t)N * z);
    u[c] = jx;
    u[plane + c] = jy;
    u[2 * plane + c] = jz;
}

// u in FP32 for storage computed in FP32, the populations of a cell added in
// their order (the fused DUGKS step forms the same sums).  SHIFTED: the LBE
// pull layout; its row offsets are formed once per cell, which with the index
// arithmetic of stored_index took as long as the loads (256^3 LBE, velocity and
// reduction together, a step with E and eps less the step: FP32 317 -> 260 us,
// FP16 330 -> 176 us with four cells a thread).
template <int I>
__device__ __forceinline__ void add_velocity(float (&j)[3], float v) {
    if constexpr (cx(I) > 0) j[0] += v;
    if constexpr (cx(I) < 0) j[0] -= v;
    if constexpr (cy(I) > 0) j[1] += v;
    if constexpr (cy(I) < 0) j[1] -= v;
    if constexpr (cz(I) > 0) j[2] += v;
    if constexpr (cz(I) < 0) j[2] -= v;
}

KIN_DEBUG_ACCESSOR(debug_word_stats)

template <typename S, bool SHIFTED>
__global__ void velocity32_kernel(const S* st, int N, size_t plane, float* __restrict__ u) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    grid_begin();
    if (x >= N) return;
    const int y = blockIdx.y, z = blockIdx.z;
    const size_t c = (size_t)x + (size_t)N * (y + (size_t)N * z);
    float f[Q];
    if constexpr (SHIFTED) {
        lbe_gather<S>(st, N, plane, x, y, z, f);
    } else {
#pragma unroll
        for (int i = 1; i < Q; ++i) f[i] = Traits<S>::load_l2(st + i * plane + c);
    }
    float j[3] = {0.0f, 0.0f, 0.0f};
    static_for<1, Q>([&](auto ic) { add_velocity<decltype(ic)::value>(j, f[decltype(ic)::value]); });
    u[c] = j[0];
    u[plane + c] = j[1];
    u[2 * plane + c] = j[2];
}

// 2-byte storage, N % 4 == 0: four x-neighbouring cells a thread, read as aligned
// 8-byte words (as the LBE step does), the same sums per cell.
template <typename S, bool SHIFTED>
__global__ void __launch_bounds__(128) velocity32v4_kernel(const S* st, int N, size_t plane, float* __restrict__ u) {
    const int x = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
    grid_begin();
    if (x >= N) return;
    const int y = blockIdx.y, z = blockIdx.z;
    unsigned w[Q][2];
    if constexpr (SHIFTED) {
        lbe_gather4p<S>(st, N, plane, x, y, z, w);
    } else {
        const size_t c = (size_t)x + (size_t)N * (y + (size_t)N * z);
#pragma unroll
        for (int i = 1; i < Q; ++i) {
            const uint2 v = __ldcg(reinterpret_cast<const uint2*>(st + i * plane + c));
            w[i][0] = v.x;
            w[i][1] = v.y;
        }
    }
    float j[4][3];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        j[k][0] = j[k][1] = j[k][2] = 0.0f;
        static_for<1, Q>([&](auto ic) {
            constexpr int I = decltype(ic)::value;
            add_velocity<I>(j[k], Half1<S>::get(w[I][k >> 1], k & 1));
        });
    }
    float* o = u + ((size_t)x + (size_t)N * (y + (size_t)N * z));
#pragma unroll
    for (int a = 0; a < 3; ++a)
        *reinterpret_cast<float4*>(o + a * plane) = make_float4(j[0][a], j[1][a], j[2][a], j[3][a]);
}

constexpr int RED_THREADS = 256;

// One cell a thread and pass (FP64 arithmetic runs at 1/64 of the FP32 rate, so
// a small box has to reach every SM: 32^3 FP64 in 16 blocks took 27 us).
int stats_blocks(int N) {
    const long long n = (long long)N * N * N;
    return (int)std::min<long long>((n + RED_THREADS - 1) / RED_THREADS, kStatsMaxBlocks);
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Sums of a and b over the block, in thread 0: warps by shuffles, then the warps'
// sums by shuffles of the first (a chain of 8 FP64 additions, each ~60 cycles).
__device__ __forceinline__ void block_sum2(double& a, double& b) {
    constexpr int W = RED_THREADS / 32;
    __shared__ double sh[2][W];
    a = warp_sum(a);
    b = warp_sum(b);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) {
        sh[0][wid] = a;
        sh[1][wid] = b;
    }
    __syncthreads();
    if (wid == 0) {
        a = sh[0][lane % W];
        b = sh[1][lane % W];
#pragma unroll
        for (int o = W / 2; o > 0; o >>= 1) {
            a += __shfl_down_sync(0xffffffffu, a, o);
            b += __shfl_down_sync(0xffffffffu, b, o);
        }
    }
}

// E = <u.u> / 2 and eps = 2 nu <s_ab s_ab> of the sums, as factors (two FP64
// divisions at the end of the reduction took 1.4 us).
struct EdScale {
    double E, eps;
};
static EdScale ed_scale(int N, double nu) {
    const double n = (double)N * N * N;
    return EdScale{0.5 / n, 2.0 * nu / n};
}

// Fixed-order sum of the block partials {sum |u|^2, sum s_ab s_ab} by one block:
// thread t takes partials t, t + RED_THREADS, ..., then block_sum2.
__device__ __forceinline__ void ed_total(const double* partial, int nblocks, const EdScale& scale, const EdSink& sink) {
    double a = 0.0, b = 0.0;
    for (int i = threadIdx.x; i < nblocks; i += RED_THREADS) {
        a += __ldcg(partial + 2 * i);
        b += __ldcg(partial + 2 * i + 1);
    }
    block_sum2(a, b);
    if (threadIdx.x == 0) {
        const double E = a * scale.E, eps = b * scale.eps;
        sink.out[0] = E;
        sink.out[1] = eps;
        if (sink.host) {
            sink.host[0] = E;
            sink.host[1] = eps;
            if (sink.err) *reinterpret_cast<int*>(sink.host + 2) = __ldcg(sink.err);
        }
    }
}

// A block's sums into its partial; the last block to get here (counter, which
// wraps to zero for the next call) forms the total.  One launch instead of two:
// the one-block total took 6 us of its own.
__device__ __forceinline__ void ed_block_done(double a, double b, double* partial, const EdScale& scale,
                                              const EdSink& sink) {
    block_sum2(a, b);
    if (threadIdx.x == 0) {
        partial[2 * blockIdx.x] = a;
        partial[2 * blockIdx.x + 1] = b;
    }
    if (!sink.counter) return;
    __shared__ bool last;
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicInc(sink.counter, gridDim.x - 1) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    ed_total(partial, gridDim.x, scale, sink);
}

// Reduction of |u|^2 and s_ab s_ab in FP64; each thread walks a fixed
// grid-stride sequence of cells.  With g_ab = u_b(+e_a) - u_b(-e_a),
// s_ab s_ab = sum_a g_aa^2 / 4 + sum_{a<b} (g_ab + g_ba)^2 / 8: 21 FP64
// operations a cell (they are what bounds the kernel), the factors exact.
__global__ void __launch_bounds__(RED_THREADS)
    ed_partial_kernel(const double* u, int N, EdScale scale, double* partial, EdSink sink) {
    grid_begin();
    const size_t n = (size_t)N * N * N;
    const double* U[3] = {u, u + n, u + 2 * n};
    double se = 0.0, sd = 0.0, so = 0.0;
    // N <= 1024: cell indices fit in 32 bits
    const unsigned un = (unsigned)N, nn = un * un;
    for (unsigned c = blockIdx.x * RED_THREADS + threadIdx.x; c < (unsigned)n; c += gridDim.x * RED_THREADS) {
        const unsigned z = c / nn, r = c - z * nn, y = r / un, x = r - y * un;
        const unsigned up[3] = {x + 1 == un ? c - x : c + 1, y + 1 == un ? c - y * un : c + un,
                                z + 1 == un ? c - z * nn : c + nn};
        const unsigned dn[3] = {x == 0 ? c + un - 1 : c - 1, y == 0 ? c + nn - un : c - un,
                                z == 0 ? c + (un - 1) * nn : c - nn};
        double g[3][3];
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) g[a][b] = U[b][up[a]] - U[b][dn[a]];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            sd = fma(g[a][a], g[a][a], sd);
            const double o = g[a][(a + 1) % 3] + g[(a + 1) % 3][a];
            so = fma(o, o, so);
            const double v = U[a][c];
            se = fma(v, v, se);
        }
    }
    ed_block_done(se, 0.25 * sd + 0.125 * so, partial, scale, sink);
}

// One cell's |u|^2 and s_ab s_ab in FP32 (the form of ed_partial_kernel), formed
// before they are added to the running sums.
__device__ __forceinline__ void add_cell(const float (&g)[3][3], const float (&u)[3], float& fe, float& fs) {
    const float d = fmaf(g[2][2], g[2][2], fmaf(g[1][1], g[1][1], g[0][0] * g[0][0]));
    const float xy = g[0][1] + g[1][0], yz = g[1][2] + g[2][1], zx = g[2][0] + g[0][2];
    const float o = fmaf(zx, zx, fmaf(yz, yz, xy * xy));
    fs += fmaf(0.5f, o, d) * 0.25f;
    fe += fmaf(u[2], u[2], fmaf(u[1], u[1], u[0] * u[0]));
}

// FP32 counterpart of ed_partial_kernel: block b takes the rows (y, z) =
// b, b + gridDim.x, ... and its threads the cells of a row; the per-cell
// |u|^2 and s_ab s_ab are formed in FP32, summed in FP32 over at most 8 rows
// and then in FP64, in a fixed order.
__global__ void __launch_bounds__(RED_THREADS)
    ed32_partial_kernel(const float* u, int N, EdScale scale, double* partial, EdSink sink) {
    grid_begin();
    const size_t n = (size_t)N * N * N;
    // component bases; offsets inside a component fit in 32 bits (N <= 1024)
    const float* U[3] = {u, u + n, u + 2 * n};
    double se = 0.0, ss = 0.0;
    float fe = 0.0f, fs = 0.0f;
    int rows_in_chunk = 0;
    for (int r = blockIdx.x; r < N * N; r += gridDim.x) {
        if (rows_in_chunk == 8) {
            se += (double)fe;
            ss += (double)fs;
            fe = fs = 0.0f;
            rows_in_chunk = 0;
        }
        ++rows_in_chunk;
        const int y = r % N, z = r / N;
        const int row = N * r;
        const int rows[3][2] = {{row, row},
                                {N * (wrap_inc(y, N) + N * z), N * (wrap_dec(y, N) + N * z)},
                                {N * (y + N * wrap_inc(z, N)), N * (y + N * wrap_dec(z, N))}};
        for (int x = threadIdx.x; x < N; x += RED_THREADS) {
            const int xs[3][2] = {{wrap_inc(x, N), wrap_dec(x, N)}, {x, x}, {x, x}};
            float g[3][3];  // g[a][b] = 2 d u_b / d x_a, central differences
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int b = 0; b < 3; ++b)
                    g[a][b] = U[b][rows[a][0] + xs[a][0]] - U[b][rows[a][1] + xs[a][1]];
            const float v[3] = {U[0][row + x], U[1][row + x], U[2][row + x]};
            add_cell(g, v, fe, fs);
        }
    }
    se += (double)fe;
    ss += (double)fs;
    ed_block_done(se, ss, partial, scale, sink);
}

// The same for N a multiple of 4, four cells per thread: a thread reads its
// four cells and their y and z neighbours as float4 and the two outer x
// neighbours as scalars, which cuts the load instructions fourfold.  Block b
// takes groups of rpi = RED_THREADS / (N/4) rows, b, b + gridDim.x, ...; the
// terms of a thread's cells are summed in cell order, in FP32 over at most 8
// row groups and then in FP64.
__global__ void __launch_bounds__(RED_THREADS)
    ed32v4_partial_kernel(const float* u, int N, EdScale scale, double* partial, EdSink sink) {
    grid_begin();
    const size_t n = (size_t)N * N * N;
    const float* U[3] = {u, u + n, u + 2 * n};
    const int gpr = N / 4, rpi = RED_THREADS / gpr;
    const int rsub = threadIdx.x / gpr, x = 4 * (threadIdx.x % gpr);
    const bool active = rsub < rpi;
    const int xm = (x == 0 ? N : x) - 1, xp = x + 4 == N ? 0 : x + 4;
    double se = 0.0, ss = 0.0;
    float fe = 0.0f, fs = 0.0f;
    int groups_in_chunk = 0;
    const int nrows = N * N;
    for (int rg = blockIdx.x; rg * rpi < nrows; rg += gridDim.x) {
        if (groups_in_chunk == 8) {
            se += (double)fe;
            ss += (double)fs;
            fe = fs = 0.0f;
            groups_in_chunk = 0;
        }
        ++groups_in_chunk;
        const int r = rg * rpi + rsub;
        if (!active || r >= nrows) continue;
        const int y = r % N, z = r / N;
        const int row = N * r;
        const int ryp = N * (wrap_inc(y, N) + N * z), rym = N * (wrap_dec(y, N) + N * z);
        const int rzp = N * (y + N * wrap_inc(z, N)), rzm = N * (y + N * wrap_dec(z, N));
        float g[4][3][3];  // g[cell][a][b] = 2 d u_b / d x_a
        float c[4][3];
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const float4 cc = *reinterpret_cast<const float4*>(U[b] + row + x);
            const float4 yp = *reinterpret_cast<const float4*>(U[b] + ryp + x);
            const float4 ym = *reinterpret_cast<const float4*>(U[b] + rym + x);
            const float4 zp = *reinterpret_cast<const float4*>(U[b] + rzp + x);
            const float4 zm = *reinterpret_cast<const float4*>(U[b] + rzm + x);
            const float l = U[b][row + xm], rr = U[b][row + xp];
            g[0][0][b] = cc.y - l;
            g[1][0][b] = cc.z - cc.x;
            g[2][0][b] = cc.w - cc.y;
            g[3][0][b] = rr - cc.z;
            g[0][1][b] = yp.x - ym.x;
            g[1][1][b] = yp.y - ym.y;
            g[2][1][b] = yp.z - ym.z;
            g[3][1][b] = yp.w - ym.w;
            g[0][2][b] = zp.x - zm.x;
            g[1][2][b] = zp.y - zm.y;
            g[2][2][b] = zp.z - zm.z;
            g[3][2][b] = zp.w - zm.w;
            c[0][b] = cc.x;
            c[1][b] = cc.y;
            c[2][b] = cc.z;
            c[3][b] = cc.w;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            add_cell(g[j], c[j], fe, fs);
        }
    }
    se += (double)fe;
    ss += (double)fs;
    ed_block_done(se, ss, partial, scale, sink);
}

__global__ void __launch_bounds__(RED_THREADS)
    ed_final_kernel(const double* partial, int nblocks, EdScale scale, EdSink sink) {
    grid_begin();
    ed_total(partial, nblocks, scale, sink);
}

cudaError_t energy_dissipation(const double* u, int N, double nu, double* partials, const EdSink& sink,
                               cudaStream_t stream) {
    const int nb = stats_blocks(N);
    cudaError_t e = launch_next(ed_partial_kernel, nb, RED_THREADS, 0, stream, u, N, ed_scale(N, nu), partials, sink);
    if (e != cudaSuccess || sink.counter) return e;
    return launch_next(ed_final_kernel, 1, RED_THREADS, 0, stream, (const double*)partials, nb, ed_scale(N, nu), sink);
}

cudaError_t energy_dissipation32(const float* u, int N, double nu, double* partials, const EdSink& sink,
                                 cudaStream_t stream) {
    if (N % 4 == 0 && N / 4 <= RED_THREADS) {
        const int rows = RED_THREADS / (N / 4);  // a block's rows at a time
        const int nb = std::min(stats_blocks(N), (N * N + rows - 1) / rows);
        return launch_next(ed32v4_partial_kernel, nb, RED_THREADS, 0, stream, u, N, ed_scale(N, nu), partials, sink);
    }
    return launch_next(ed32_partial_kernel, std::min(stats_blocks(N), N * N), RED_THREADS, 0, stream, u, N,
                       ed_scale(N, nu), partials, sink);
}

// ---------------------------------------------------------------------------
// Spectrum shells.  Modes of the half-complex layout [kz][ky][kx],
// kx = 0..N/2; a mode with 0 < kx < N/2 also stands for its conjugate.
// Lanes of a warp that fall in the same shell are summed in lane order by the
// lowest lane, which adds the result to a warp-private shell array; the block
// then adds its warps' arrays in warp order.
constexpr int SPEC_THREADS = 256;

int spectrum_blocks(int N) {
    long long n = (long long)N * N * (N / 2 + 1);
    long long b = (n + SPEC_THREADS * 16 - 1) / (SPEC_THREADS * 16);
    if (b > 304) b = 304;
    if (b < 1) b = 1;
    return (int)b;
}

// CT: double2 (FP64 transform) or float2 (FP32 transform, |u_hat|^2 formed
// in FP32 and summed in FP64).
template <typename CT>
__global__ void __launch_bounds__(SPEC_THREADS)
    shell_partial_kernel(const CT* __restrict__ u0, const CT* __restrict__ u1,
                         const CT* __restrict__ u2, int N, int nshell, double scale,
                         int weight_n2, double* __restrict__ partial) {
    extern __shared__ double bins[];  // [SPEC_THREADS/32][nshell]
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    double* mybins = bins + wid * nshell;
    for (int s = lane; s < nshell; s += 32) mybins[s] = 0.0;
    __syncwarp();
    __shared__ double xch[SPEC_THREADS];  // lane values for the shell sums
    const int nh = N / 2 + 1;
    const int nmode = N * N * nh;  // < 2^31 for N <= 1024
    // each warp handles consecutive chunks of 32 modes
    const int nwarps = gridDim.x * (SPEC_THREADS / 32);
    const int gw = blockIdx.x * (SPEC_THREADS / 32) + wid;
    for (int base = gw * 32; base < nmode; base += nwarps * 32) {
        const int m = base + lane;
        int shell = -1;
        double e = 0.0;
        if (m < nmode) {
            const int kx = m % nh, t = m / nh;
            const int ky = t % N, kz = t / N;
            const int sy = ky > N / 2 ? ky - N : ky;
            const int sz = kz > N / 2 ? kz - N : kz;
            const int n2 = kx * kx + sy * sy + sz * sz;  // < 2^24: exact in FP32
            // nearest integer to |n|; |n| is never within FP32 rounding of a half-integer
            shell = (int)floorf(sqrtf((float)n2) + 0.5f);
            const CT a = u0[m], b = u1[m], c = u2[m];
            const double amp = (double)((a.x * a.x + a.y * a.y) + (b.x * b.x + b.y * b.y) + (c.x * c.x + c.y * c.y));
            const double w = (kx > 0 && 2 * kx < N) ? 2.0 : 1.0;
            e = amp * (weight_n2 ? (double)n2 * w : w);
        }
        const unsigned same = __match_any_sync(0xffffffffu, shell);
        const int leader = __ffs(same) - 1;
        xch[threadIdx.x] = e;
        __syncwarp();
        if (lane == leader && shell >= 0 && shell < nshell) {
            // the lanes of this shell in lane order
            double acc = 0.0;
            for (unsigned msk = same; msk; msk &= msk - 1) acc += xch[wid * 32 + __ffs(msk) - 1];
            mybins[shell] += acc;
        }
        __syncwarp();
    }
    __syncthreads();
    for (int s = threadIdx.x; s < nshell; s += SPEC_THREADS) {
        double a = 0.0;
        for (int w = 0; w < SPEC_THREADS / 32; ++w) a += bins[w * nshell + s];
        partial[(size_t)blockIdx.x * nshell + s] = a * scale;
    }
}

__global__ void shell_final_kernel(const double* __restrict__ partial, int nblocks, int nshell,
                                   double* __restrict__ out) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= nshell) return;
    double a = 0.0;
    for (int b = 0; b < nblocks; ++b) a += partial[(size_t)b * nshell + s];
    out[s] = a;
}

// ---------------------------------------------------------------------------
// Spectral derivative d_a u_a of one component: u_hat (half-complex, unscaled
// D2Z output) times i k_a / N^3, the Nyquist wavenumber of axis a set to zero;
// the Z2D of the result is the derivative field.
// k1 = 2 pi / N / N^3 (formed on the host: a division a mode cost as much as the
// memory traffic).
__global__ void deriv_mult_kernel(double2* __restrict__ uh, int N, int axis, double k1) {
    const int nh = N / 2 + 1;
    const int kx = blockIdx.x * blockDim.x + threadIdx.x;
    if (kx >= nh) return;
    const int ky = blockIdx.y, kz = blockIdx.z;
    const size_t m = (size_t)kx + (size_t)nh * (ky + (size_t)N * kz);
    int n = axis == 0 ? kx : axis == 1 ? ky : kz;
    if (axis != 0 && n > N / 2) n -= N;
    const bool nyquist = (N % 2 == 0) && (n == N / 2 || n == -N / 2);
    const double k = nyquist ? 0.0 : (double)n * k1;
    const double2 v = uh[m];
    uh[m] = make_double2(-k * v.y, k * v.x);
}

constexpr int MOM_THREADS = 256;

// Block partials of sum d^2, d^3, d^4 for the three derivative fields d_a
// (fixed grid-stride order, then warp and block order): partial[9 b + 3 a + p].
__global__ void __launch_bounds__(MOM_THREADS)
    deriv_moments_kernel(const double* __restrict__ d, int N, double* __restrict__ partial) {
    const size_t n = (size_t)N * N * N;
    double acc[9];
#pragma unroll
    for (int j = 0; j < 9; ++j) acc[j] = 0.0;
    for (size_t c = (size_t)blockIdx.x * MOM_THREADS + threadIdx.x; c < n; c += (size_t)gridDim.x * MOM_THREADS) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const double v = d[a * n + c], v2 = v * v;
            acc[3 * a] += v2;
            acc[3 * a + 1] += v2 * v;
            acc[3 * a + 2] += v2 * v2;
        }
    }
    __shared__ double sh[9][MOM_THREADS / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int j = 0; j < 9; ++j) {
        const double w = warp_sum(acc[j]);
        if (lane == 0) sh[j][wid] = w;
    }
    __syncthreads();
    if (threadIdx.x < 9) {
        double t = 0.0;
        for (int w = 0; w < MOM_THREADS / 32; ++w) t += sh[threadIdx.x][w];
        partial[9 * (size_t)blockIdx.x + threadIdx.x] = t;
    }
}

__global__ void deriv_moments_final_kernel(const double* __restrict__ partial, int nblocks, size_t n,
                                           double* __restrict__ out) {
    const int j = threadIdx.x;
    if (j >= 9) return;
    double t = 0.0;
    for (int b = 0; b < nblocks; ++b) t += partial[9 * (size_t)b + j];
    out[j] = t / (double)n;
}

int deriv_moment_blocks(int N) {
    long long n = (long long)N * N * N;
    long long b = (n + MOM_THREADS * 16 - 1) / (MOM_THREADS * 16);
    if (b > 608) b = 608;
    if (b < 1) b = 1;
    return (int)b;
}

cudaError_t derivative_multiply(double2* uh, int N, int axis, cudaStream_t stream) {
    const int nh = N / 2 + 1;
    const int bx = nh < 128 ? ((nh + 31) / 32) * 32 : 128;
    dim3 g((nh + bx - 1) / bx, N, N);
    const double k1 = 2.0 * 3.14159265358979323846 / N / ((double)N * N * N);
    deriv_mult_kernel<<<g, bx, 0, stream>>>(uh, N, axis, k1);
    return cudaGetLastError();
}

cudaError_t derivative_moments(const double* d, int N, double* partial, double* out, cudaStream_t stream) {
    const int nb = deriv_moment_blocks(N);
    deriv_moments_kernel<<<nb, MOM_THREADS, 0, stream>>>(d, N, partial);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    deriv_moments_final_kernel<<<1, 32, 0, stream>>>(partial, nb, (size_t)N * N * N, out);
    return cudaGetLastError();
}

template <typename CT>
static cudaError_t spectrum_shells_t(const void* uh0, const void* uh1, const void* uh2, int N, int nshell,
                                     double inv, int weight_n2, double* partial, double* out,
                                     cudaStream_t stream) {
    const int nb = spectrum_blocks(N);
    const size_t smem = sizeof(double) * nshell * (SPEC_THREADS / 32);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(shell_partial_kernel<CT>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    shell_partial_kernel<CT><<<nb, SPEC_THREADS, smem, stream>>>(
        (const CT*)uh0, (const CT*)uh1, (const CT*)uh2, N, nshell, 0.5 * inv * inv, weight_n2, partial);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    shell_final_kernel<<<(nshell + 127) / 128, 128, 0, stream>>>(partial, nb, nshell, out);
    return cudaGetLastError();
}

cudaError_t spectrum_shells(const void* uh0, const void* uh1, const void* uh2, int N, int nshell,
                            double inv, int weight_n2, double* partial, double* out,
                            cudaStream_t stream) {
    return spectrum_shells_t<double2>(uh0, uh1, uh2, N, nshell, inv, weight_n2, partial, out, stream);
}

cudaError_t spectrum_shells32(const void* uh0, const void* uh1, const void* uh2, int N, int nshell,
                              double inv, double* partial, double* out, cudaStream_t stream) {
    return spectrum_shells_t<float2>(uh0, uh1, uh2, N, nshell, inv, 0, partial, out, stream);
}

// ---------------------------------------------------------------------------
// f = f_eq(0, u) in the storage's compute type: FP64 for FP64 storage, FP32
// otherwise (FP64 arithmetic on this GPU runs at a small fraction of the FP32
// rate, and an FP32-stored state needs no more than FP32 arithmetic).
template <typename S>
__global__ void feq_kernel(const double* __restrict__ u, bool shifted, int N, size_t plane,
                           S* __restrict__ st) {
    using C = typename Traits<S>::C;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= N) return;
    const int y = blockIdx.y, z = blockIdx.z;
    const size_t c = (size_t)x + (size_t)N * (y + (size_t)N * z);
    const C ux = (C)u[c], uy = (C)u[plane + c], uz = (C)u[2 * plane + c];
    const C usq15 = C(1.5) * (ux * ux + uy * uy + uz * uz);
    static_for<0, Q>([&](auto ic) {
        constexpr int I = decltype(ic)::value;
        Traits<S>::store(st + I * plane + stored_index<I>(x, y, z, N, shifted), feq_i<I>(C(0), ux, uy, uz, usq15));
    });
}

template <typename S>
__global__ void set_pop_kernel(int i, const double* __restrict__ pl, bool shifted, int N,
                               size_t plane, S* __restrict__ st) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= N) return;
    const int y = blockIdx.y, z = blockIdx.z;
    const size_t c = (size_t)x + (size_t)N * (y + (size_t)N * z);
    Traits<S>::store(st + i * plane + stored_index_rt(i, x, y, z, N, shifted),
                     (typename Traits<S>::C)pl[c]);
}

template <typename S>
__global__ void get_pop_kernel(int i, const S* __restrict__ st, bool shifted, int N, size_t plane,
                               double* __restrict__ pl) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= N) return;
    const int y = blockIdx.y, z = blockIdx.z;
    const size_t c = (size_t)x + (size_t)N * (y + (size_t)N * z);
    pl[c] = (double)Traits<S>::load(st + i * plane + stored_index_rt(i, x, y, z, N, shifted));
}

template <typename S>
__global__ void sample_kernel(const S* __restrict__ st, bool shifted, int N, size_t plane,
                              const int64_t* __restrict__ cells, int64_t n, double* __restrict__ out) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n * Q) return;
    const int64_t k = t / Q;
    const int i = (int)(t % Q);
    const int64_t c = cells[k];
    const int x = (int)(c % N), y = (int)((c / N) % N), z = (int)(c / ((int64_t)N * N));
    out[t] = (double)Traits<S>::load(st + i * plane + stored_index_rt(i, x, y, z, N, shifted));
}

// delta-rho of every cell (Eq. 8) into prev (mode 0), or (mode 1) the largest
// |delta-rho - prev| over the box into *maxbits as the bits of a
// non-negative float (ordered like the values, so atomicMax applies).
template <typename S>
__global__ void drho_change_kernel(const S* __restrict__ st, bool shifted, int N, size_t plane,
                                   double* __restrict__ prev, unsigned* maxbits, int mode) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y, z = blockIdx.z;
    float d = 0.0f;
    if (x < N) {
        double rho = 0.0;
        static_for<0, Q>([&](auto ic) {
            constexpr int I = decltype(ic)::value;
            rho += (double)Traits<S>::load(st + I * plane + stored_index<I>(x, y, z, N, shifted));
        });
        const size_t c = (size_t)x + (size_t)N * (y + (size_t)N * z);
        if (mode == 0) prev[c] = rho;
        else d = (float)fabs(rho - prev[c]);
    }
    if (mode == 1) {
        for (int o = 16; o > 0; o >>= 1) d = fmaxf(d, __shfl_down_sync(0xffffffffu, d, o));
        if ((threadIdx.x & 31) == 0) atomicMax(maxbits, __float_as_uint(d));
    }
}

__global__ void nonfinite_kernel(const double* __restrict__ v, size_t n, int* flag) {
    bool bad = false;
    for (size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x; k < n;
         k += (size_t)gridDim.x * blockDim.x)
        bad |= !isfinite(v[k]);
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(flag, 1);
}

static dim3 row_grid(int N, int& bx) {
    bx = N >= 128 ? 128 : ((N + 31) / 32) * 32;
    return dim3((N + bx - 1) / bx, N, N);
}

#define KIN_DISPATCH(storage, CALL)                       \
    switch (storage) {                                    \
        case ST_F32: { using S = float; CALL; } break;    \
        case ST_F16: { using S = __half; CALL; } break;   \
        case ST_BF16: { using S = __nv_bfloat16; CALL; } break; \
        case ST_F64: { using S = double; CALL; } break;   \
        default: return cudaErrorInvalidValue;            \
    }

cudaError_t velocity_field(int storage, const void* state, bool shifted, int N, double* u,
                           cudaStream_t stream) {
    int bx;
    dim3 g = row_grid(N, bx);
    const size_t plane = (size_t)N * N * N;
    KIN_DISPATCH(storage, return launch_next(velocity_kernel<S>, g, bx, 0, stream, (const S*)state, shifted, N, plane, u));
    return cudaSuccess;
}

template <typename S, bool SHIFTED>
static cudaError_t velocity32_t(const void* state, int N, float* u, cudaStream_t stream) {
    const size_t plane = (size_t)N * N * N;
    if constexpr (sizeof(S) == 2) {
        if (N % 4 == 0) {
            const int nv = N / 4, bx = nv >= 64 ? 64 : 32;
            return launch_next(velocity32v4_kernel<S, SHIFTED>, dim3((nv + bx - 1) / bx, N, N), bx, 0, stream,
                               (const S*)state, N, plane, u);
        }
    }
    int bx;
    const dim3 g = row_grid(N, bx);
    return launch_next(velocity32_kernel<S, SHIFTED>, g, bx, 0, stream, (const S*)state, N, plane, u);
}

cudaError_t velocity_field32(int storage, const void* state, bool shifted, int N, float* u,
                             cudaStream_t stream) {
    switch (storage) {
        case ST_F32: return shifted ? velocity32_t<float, true>(state, N, u, stream) : velocity32_t<float, false>(state, N, u, stream);
        case ST_F16: return shifted ? velocity32_t<__half, true>(state, N, u, stream) : velocity32_t<__half, false>(state, N, u, stream);
        case ST_BF16:
            return shifted ? velocity32_t<__nv_bfloat16, true>(state, N, u, stream)
                           : velocity32_t<__nv_bfloat16, false>(state, N, u, stream);
    }
    return cudaErrorInvalidValue;
}

cudaError_t equilibrium_from_velocity(int storage, const double* u, bool shifted, int N,
                                      void* state, cudaStream_t stream) {
    int bx;
    dim3 g = row_grid(N, bx);
    const size_t plane = (size_t)N * N * N;
    KIN_DISPATCH(storage, (feq_kernel<S><<<g, bx, 0, stream>>>(u, shifted, N, plane, (S*)state)));
    return cudaGetLastError();
}

cudaError_t set_population(int storage, int i, const double* pl, bool shifted, int N, void* state,
                           cudaStream_t stream) {
    int bx;
    dim3 g = row_grid(N, bx);
    const size_t plane = (size_t)N * N * N;
    KIN_DISPATCH(storage, (set_pop_kernel<S><<<g, bx, 0, stream>>>(i, pl, shifted, N, plane, (S*)state)));
    return cudaGetLastError();
}

cudaError_t get_population(int storage, int i, const void* state, bool shifted, int N, double* pl,
                           cudaStream_t stream) {
    int bx;
    dim3 g = row_grid(N, bx);
    const size_t plane = (size_t)N * N * N;
    KIN_DISPATCH(storage, (get_pop_kernel<S><<<g, bx, 0, stream>>>(i, (const S*)state, shifted, N, plane, pl)));
    return cudaGetLastError();
}

cudaError_t sample_cells(int storage, const void* state, bool shifted, int N, const int64_t* cells,
                         int64_t n, double* out, cudaStream_t stream) {
    if (n <= 0) return cudaSuccess;
    const size_t plane = (size_t)N * N * N;
    const int64_t tot = n * Q;
    const int threads = 256;
    const unsigned blocks = (unsigned)((tot + threads - 1) / threads);
    KIN_DISPATCH(storage, (sample_kernel<S><<<blocks, threads, 0, stream>>>((const S*)state, shifted, N, plane, cells, n, out)));
    return cudaGetLastError();
}

cudaError_t scan_nonfinite(const double* v, size_t n, int* flag, cudaStream_t stream) {
    nonfinite_kernel<<<304, 256, 0, stream>>>(v, n, flag);
    return cudaGetLastError();
}

cudaError_t drho_change(int storage, const void* state, bool shifted, int N, double* prev, unsigned* maxbits,
                        int mode, cudaStream_t stream) {
    int bx;
    dim3 g = row_grid(N, bx);
    const size_t plane = (size_t)N * N * N;
    KIN_DISPATCH(storage, (drho_change_kernel<S><<<g, bx, 0, stream>>>((const S*)state, shifted, N, plane, prev,
                                                                      maxbits, mode)));
    return cudaGetLastError();
}

}  // namespace kin

// ---------------------------------------------------------------------------
// E / eps reduction that allocates nothing.
//
// Some callers cannot let the library allocate device memory: a real-time
// loop must not call cudaMalloc or cudaFree (either can synchronise the whole
// device), and an application may have reserved all device memory for its own
// allocator (a framework's caching allocator, a fixed arena).  For them the
// per-block partial sums of the reduction live in this fixed array compiled
// into the library instead of in memory allocated per simulation.  It holds
// 2 x kStatsMaxBlocks doubles (19,456 bytes) and exists on every device that loads the
// library until the process exits.  Every call shares it and overwrites the
// partials it uses before reading them (nothing has to start at zero); calls
// whose kernels overlap on the GPU race on it.
namespace {

constexpr int kNoallocMaxBlocks = kin::kStatsMaxBlocks;
constexpr int kNoallocMaxN = 1024;
static_assert(kNoallocMaxBlocks >= kin::kStatsMaxBlocks, "partials must cover stats_blocks() for every N");

static __device__ __align__(256) double g_noalloc_partials[2 * kNoallocMaxBlocks];

// Device address of the array in the current device's context.  Looked up on
// every call, not cached: after a context reset the module is loaded again and
// the array may sit elsewhere.
double* noalloc_scratch(cudaError_t* err) {
    void* p = nullptr;
    *err = cudaGetSymbolAddress(&p, g_noalloc_partials);
    return *err == cudaSuccess ? (double*)p : nullptr;
}

}  // namespace

extern "C" int kin_energy_dissipation_noalloc(const double* u, int N, double nu, double* out,
                                              void* stream) {
    using namespace kin;
    if (!u || !out) return set_error(KIN_EINVAL, "NULL device pointer");
    if (N < 2 || N > kNoallocMaxN)
        return set_error(KIN_EINVAL,
                         "N = %d outside [2, %d], the sizes the fixed scratch of this entry point covers",
                         N, kNoallocMaxN);
    if (!(nu >= 0.0)) return set_error(KIN_EINVAL, "nu must be >= 0");
    const int nb = stats_blocks(N);
    if (nb > kNoallocMaxBlocks)
        return set_error(KIN_EINVAL, "reduction needs %d blocks, fixed scratch holds %d", nb,
                         kNoallocMaxBlocks);
    cudaError_t e;
    double* partials = noalloc_scratch(&e);
    if (!partials) return set_error(KIN_ECUDA, "cudaGetSymbolAddress: %s", cudaGetErrorString(e));
    EdSink sink;
    sink.out = out;  // no counter: overlapping calls would leave it set
    e = energy_dissipation(u, N, nu, partials, sink, (cudaStream_t)stream);
    if (e != cudaSuccess) return set_error(KIN_ECUDA, "reduction launch: %s", cudaGetErrorString(e));
    return KIN_OK;
}

