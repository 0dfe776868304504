// Two MRT-LBE steps in one pass over memory (FP32 storage).
//
// The step is bound by DRAM: every population is read and written once a step,
// 152 bytes a node.  Here a thread block marches along z over tiles of 30 x TY
// nodes: it relaxes every node of the tile and of a one-node rim (step t), keeps
// the post-collision populations of the planes around the current one in shared
// memory, and relaxes the tile's nodes again from there (step t + 1), so the state
// crosses DRAM once per two steps.  A population that moves up or down stays in
// its own thread's registers when it does not move across x or y.  One barrier a
// plane: what a plane writes is kept apart from what the plane before still reads
// (four, three and two slots for the upward, in-plane and downward
// populations).  Both steps use the node arithmetic of lbe_node, so the results
// are bitwise those of two single steps.
//
// 256^3: 515 us for two steps (257 a step) against 2 x 366 us, which is the copy
// roof; 2.56 GB of DRAM traffic a pair = 4.97 TB/s, issue 70 %.  6-row tiles, three
// 8-warp blocks an SM at 80 registers; two of 10 rows are level, one of 22 rows or
// blocks without the prefetch of the next plane (64 registers) are slower (270,
// 332).  Packed FP32x2 pair sums left it unchanged.
#pragma once

#include "kin_launch.cuh"
#include "lbe_node.cuh"

namespace kin {

// Slots of the populations that move across x or y, by the plane they reach:
// next (xi_z = +1), the same, the previous.
__host__ __device__ constexpr int lbe_slot(int i, int zc) {
    int n = 0;
    for (int q = 0; q < i; ++q)
        if (cz(q) == zc && (cx(q) != 0 || cy(q) != 0)) ++n;
    return n;
}
__host__ __device__ constexpr bool lbe_moves(int i) { return cx(i) != 0 || cy(i) != 0; }

// Shared memory, in floats: [slot][population][row][lane], every access of a
// thread one base address plus a constant and its slot.
template <int TY>
struct LbePairSmem {
    static constexpr int ROWS = TY + 2, POP = ROWS * 32;
    // planes k - 2 .. k + 1 of the 4 upward populations, k - 1 .. k + 1 of the 8
    // in-plane ones, k and k + 1 of the 4 downward ones: what is written for
    // plane k + 1 is apart from what plane k's update still reads
    static constexpr int UP = 4, FLAT = UP + 4 * 4 * POP, DOWN = FLAT + 3 * 8 * POP, FLOATS = DOWN + 2 * 4 * POP + 4;
};

constexpr int kPairRows = 6, kPairBlocks = 3;  // rows of a tile, blocks of an SM

template <int TY>
__global__ void __launch_bounds__(32 * (TY + 2), kPairBlocks)
    lbe_pair_kernel(const float* src, float* dst, int N, size_t plane, int zchunk, MrtRates<float> rates) {
    using SM = LbePairSmem<TY>;
    extern __shared__ __align__(16) float smem_f[];
    const int lane = threadIdx.x, row = threadIdx.y;
    const int z0 = blockIdx.z * zchunk, zend = min(z0 + zchunk, N);
    const int xr = blockIdx.x * 30 - 1 + lane, yr = blockIdx.y * TY - 1 + row;
    const int x = xr < 0 ? xr + N : xr % N, y = yr < 0 ? yr + N : yr % N;
    const bool yin = row >= 1 && row <= TY;
    const bool valid = yin && lane >= 1 && lane <= 30 && xr < N && yr < N;
    const int xo[3] = {wrap_dec(x, N), x, wrap_inc(x, N)};
    const int yo[3] = {wrap_dec(y, N) * N, y * N, wrap_inc(y, N) * N};
    const int nn = N * N, n3 = nn * N;  // N <= 1024
    float* const own = smem_f + row * 32 + lane;
    grid_begin();
    (void)KIN_CHECK(row < SM::ROWS && lane < 32, DBG_LBE_SLOT, row * 64 + lane);

    // plane offsets of planes k - 1, k, k + 1 of the next load (N >= 2)
    int zo[3];
    zo[0] = (z0 >= 2 ? z0 - 2 : z0 - 2 + N) * nn;
    zo[1] = zo[0] + nn == n3 ? 0 : zo[0] + nn;
    zo[2] = zo[1] + nn == n3 ? 0 : zo[1] + nn;
    float f[Q];
    auto load = [&] {
        static_for<0, Q>([&](auto ic) {
            constexpr int I = decltype(ic)::value;
            const int idx = xo[1 - cx(I)] + yo[1 - cy(I)] + zo[1 - cz(I)];
            if (!KIN_CHECK(idx >= 0 && (size_t)idx < plane, DBG_LBE_LOAD, idx)) f[I] = 0.0f;
            else f[I] = __ldcg(src + (size_t)I * plane + idx);
        });
        zo[0] = zo[1];
        zo[1] = zo[2];
        zo[2] = zo[2] + nn == n3 ? 0 : zo[2] + nn;
    };

    float rest = 0.0f, z5a = 0.0f, z5b = 0.0f;  // f_0 of plane k - 1, f_5 of planes k - 1 and k - 2
    int up = 0, flat = 0, down = 0;              // offsets of plane k's slots
    int flat_before = 0, up_before = 0;          // of plane k - 1's in-plane and plane k - 2's upward slot
    int up_last = 0;
    load();
    for (int k = z0 - 1; k <= zend; ++k) {
        mrt_collide_as<float, false>(f, rates);
        static_for<0, Q>([&](auto ic) {
            constexpr int I = decltype(ic)::value;
            if constexpr (lbe_moves(I)) {
                constexpr int O = lbe_slot(I, cz(I)) * SM::POP;
                if constexpr (cz(I) > 0) own[SM::UP + O + up] = f[I];
                if constexpr (cz(I) == 0) own[SM::FLAT + O + flat] = f[I];
                if constexpr (cz(I) < 0) own[SM::DOWN + O + down] = f[I];
            }
        });
        const float f0 = f[0], f5 = f[5], f6 = f[6];
        if (k < zend) load();
        __syncthreads();
        if (k > z0 && yin) {
            // the slots' first words; a row, and a word beside it, each way is inside (yin)
            (void)KIN_CHECK(up >= 0 && up < SM::FLAT - SM::UP && up_before >= 0 && up_before < SM::FLAT - SM::UP &&
                                flat >= 0 && flat < SM::DOWN - SM::FLAT && flat_before >= 0 &&
                                flat_before < SM::DOWN - SM::FLAT && down >= 0 && down < 8 * SM::POP,
                            DBG_LBE_SLOT, up);
            float g[Q];
            g[0] = rest;
            g[5] = z5b;
            g[6] = f6;
            static_for<0, Q>([&](auto ic) {
                constexpr int I = decltype(ic)::value;
                if constexpr (lbe_moves(I)) {
                    constexpr int O = lbe_slot(I, cz(I)) * SM::POP - cy(I) * 32 - cx(I);
                    if constexpr (cz(I) > 0) g[I] = own[SM::UP + O + up_before];
                    if constexpr (cz(I) == 0) g[I] = own[SM::FLAT + O + flat_before];
                    if constexpr (cz(I) < 0) g[I] = own[SM::DOWN + O + down];
                }
            });
            mrt_collide_as<float, false>(g, rates);
            if (valid) {
                const int c = x + y * N + (k - 1) * nn;
                if (KIN_CHECK(c >= 0 && (size_t)c < plane, DBG_LBE_STORE, c)) {
#pragma unroll
                    for (int i = 0; i < Q; ++i) __stcg(dst + (size_t)i * plane + c, g[i]);
                }
            }
        }
        z5b = z5a;
        z5a = f5;
        rest = f0;
        up_before = up_last;
        up_last = up;
        flat_before = flat;
        up = up == 3 * 4 * SM::POP ? 0 : up + 4 * SM::POP;
        flat = flat == 2 * 8 * SM::POP ? 0 : flat + 8 * SM::POP;
        down = 4 * SM::POP - down;
    }
}

// Two steps of a box of at most 32 (FP32, FP16 or BF16 storage): such a step is
// latency, not bytes (32^3: 3.5 us, of which ~1.7 are the hand-over from one grid
// to the next; in pairs 1.4 us a step).  A warp holds a whole periodic row, a block TY rows and TZ planes
// with a rim of one, one node a thread: every thread relaxes its node, the inner
// ones again from shared memory.  Most of the first step is done by several
// blocks, which costs less than a second launch.
template <typename S, int TY, int TZ>
__global__ void __launch_bounds__(32 * (TY + 2) * (TZ + 2), 1)
    lbe_small_pair_kernel(const S* src, S* dst, int N, size_t plane, MrtRates<float> rates) {
    constexpr int ROWS = TY + 2, PLANES = TZ + 2;
    extern __shared__ __align__(16) float smem_f[];  // [population][plane][row][lane]
    const int lane = threadIdx.x, row = threadIdx.y, pl = threadIdx.z;
    const int yr = blockIdx.x * TY - 1 + row, zr = blockIdx.y * TZ - 1 + pl;
    const int x = min(lane, N - 1), y = (yr + N) % N, z = (zr + N) % N;
    grid_begin();
    float f[Q];
    lbe_gather<S>(src, N, plane, x, y, z, f);
    mrt_collide_as<S, false>(f, rates);
    // what storing the state and reading it back gives
#pragma unroll
    for (int i = 0; i < Q; ++i) f[i] = (float)S(f[i]);
    constexpr int POP = PLANES * ROWS * 32;
    const int at = (pl * ROWS + row) * 32;
#pragma unroll
    for (int i = 1; i < Q; ++i) smem_f[i * POP + at + lane] = f[i];
    __syncthreads();
    if (row < 1 || row > TY || pl < 1 || pl > TZ || lane >= N || yr >= N || zr >= N) return;
    const int xs[3] = {wrap_dec(lane, N), lane, wrap_inc(lane, N)};
    static_for<1, Q>([&](auto ic) {
        constexpr int I = decltype(ic)::value;
        const int idx = I * POP + at - (cz(I) * ROWS + cy(I)) * 32 + xs[1 - cx(I)];
        if (KIN_CHECK(idx >= I * POP && idx < (I + 1) * POP, DBG_LBE_SLOT, idx)) f[I] = smem_f[idx];
    });
    mrt_collide_as<S, false>(f, rates);
    lbe_scatter<S>(dst, N, plane, lane, yr, zr, f);
}

}  // namespace kin
