// Ensemble of independent simulations advanced together by one CUDA graph
// launch per kin_ensemble_step call.
//
// DUGKS members: one persistent, cooperative kernel runs all their steps.  The
// work of one time step is a list of items (member, tile) of the fused step
// (dugks_tile.cuh).  Thread blocks take (step, item) pairs one at a time from
// a global counter, all items of step s before any of step s + 1.  A member's
// step s may start only when all its tiles of step s - 1 are done: each
// finished tile adds one to the member's counter with a GPU-scope release, and
// a block waits for count >= s * tiles with acquire loads before touching the
// member.  Every item a wait depends on was handed out earlier to a running
// block, so every wait is eventually satisfied whether or not all blocks are
// resident; it is nevertheless bounded in time and sets a status word (and
// releases every other waiter) if it runs out.
//
// LBE members: one batched launch per step covers every LBE member of a
// storage type (a block takes consecutive nodes of one member), on a second
// stream of the same graph.  The two kernels never wait on each other;
// consecutive LBE steps are ordered by their stream.  Two persistent blocks of
// 5-row tiles fill an SM's registers, so the LBE launches get the SMs before or
// after them: for the 24-member reference mix 0.347 ms a step of the DUGKS
// members plus 0.139 ms of the LBE members, 0.485 together.  Tiles that leave
// registers for LBE blocks beside them overlap and are still slower (one block
// of 7-row tiles at 160 registers: 0.601 together, where these took 0.502).
//
// Which block runs an item does not change what it computes: a member's
// results are bitwise those of stepping it alone.
//
// Double buffering: step s reads buf[(cur + s) & 1] and writes the other
// buffer; the member barrier (DUGKS) or the stream order (LBE) makes every
// read of step s - 1 precede every write of step s + 1 to the same buffer.
#include "dugks_tile.cuh"
#include "dugks_tile16.cuh"
#include "kin.h"
#include "kin_internal.h"
#include "kin_sim.h"
#include "lbe_node.cuh"

#include <nvtx3/nvToolsExt.h>

#include <algorithm>
#include <cmath>
#include <climits>
#include <cstddef>
#include <map>
#include <vector>

namespace kin {

// DUGKS member of the persistent kernel
struct EnsMember {
    void* buf[2];
    int N, storage, cur, ntiles;
    int tiles_x, tiles_y, zchunk;
    DugksCoef<float> coef;
};

// LBE member of the batched launch of its storage type
struct LbeMember {
    void* buf[2];
    int N, cur, V;    // V consecutive cells a thread (as the standalone LBE step)
    unsigned block0;  // its first block in the batched grid
    MrtRates<float> rates;
};

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void red_release_add(unsigned* p, unsigned v) {
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ int ld_relaxed(const int* p) {
    int v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Storage types of the DUGKS members of a kernel: one, or any mixture.  A kernel of
// its own for each, since three tiles in one body spill where the registers of a block
// are capped (8 rows: 664 bytes; one 2-byte type: none.  Four 64^3 FP16 members, 16
// planes: 184 against 100 us a step).
enum { HAS_F32 = 1, HAS_F16 = 2, HAS_BF16 = 4, HAS_MIXED = 7 };

// Warps of a block and rows of its FP32 tiles at tile height ty.  A 2-byte tile has a
// warp for each of its two halo rows, an FP32 tile one for both: in a kernel that
// runs 2-byte members the block holds their ty rows, and FP32 tiles of one row more.
constexpr int block_warps(int ty, int has) { return has == HAS_F32 ? ty + 1 : ty + 2; }
constexpr int rows32(int ty, int has) { return block_warps(ty, has) - 1; }

// Blocks an SM that the registers of a thread are held to.
constexpr int blocks_an_sm(int ty, int has) { return ty <= 5 && has == HAS_F32 ? 2 : 1; }

// One fused-DUGKS tile t of member M at buffer parity par.
template <typename S, int TY, int HAS>
__device__ __forceinline__ void ensemble_tile(const EnsMember& M, int par, int t, unsigned char* smem_raw) {
    const int per = M.tiles_x * M.tiles_y;
    const int bz = t / per, r = t % per;
    // a local copy of the member's coefficients: passed as a reference into
    // the member table in global memory, the items ran 13 % slower
    const DugksCoef<float> kc = M.coef;
    const S* src = static_cast<const S*>(M.buf[par]);
    S* dst = static_cast<S*>(M.buf[par ^ 1]);
    if constexpr (sizeof(S) == 2)
        two_byte::dugks_tile<S, TY>(src, dst, M.N, r % M.tiles_x, r / M.tiles_x, bz, M.zchunk, kc, smem_raw);
    else
        dugks_tile<S, rows32(TY, HAS)>(src, dst, M.N, r % M.tiles_x, r / M.tiles_x, bz, M.zchunk, kc, smem_raw);
}

// The tile as a function of its own: in the mixed kernel of 8-row tiles it spills at
// most 268 bytes (64^3: 3 FP32, 2 FP16 members and 48^3 BF16 beside LBE, 64 planes: 297
// -> 237 us a step).
template <typename S, int TY, int HAS>
__device__ __noinline__ void called_tile(const EnsMember& M, int par, int t, unsigned char* smem_raw) {
    ensemble_tile<S, TY, HAS>(M, par, t, smem_raw);
}

template <int TY, int HAS>
__device__ __forceinline__ void ensemble_body(const EnsMember* __restrict__ mem, const int2* __restrict__ items,
                                              int nitems, int nsteps, unsigned* done, unsigned* next_item,
                                              int* status, long long wait_cycles, int stall_test) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_abort;
    __shared__ unsigned s_idx;
    const int tid = threadIdx.y * 32 + threadIdx.x;
    // Blocks take (step, item) pairs in order from a global counter: every
    // item of step s is handed out before any of step s + 1, so an item only
    // waits on items already running in resident blocks.
    const unsigned total = (unsigned)nsteps * (unsigned)nitems;
    for (;;) {
        if (tid == 0) s_idx = atomicAdd(next_item, 1u);
        __syncthreads();
        const unsigned idx = s_idx;
        if (idx >= total) return;
        {
            const int s = (int)(idx / (unsigned)nitems), it = (int)(idx % (unsigned)nitems);
            const int2 item = items[it];
            const EnsMember& M = mem[item.x];
            if (tid == 0) {
                int abort = ld_relaxed(status) != 0;
                // stall_test raises the target of step 1 beyond reach, to
                // exercise the bounded wait
                const unsigned target = (unsigned)s * (unsigned)M.ntiles + (stall_test && s == 1 ? 1u : 0u);
                if (!abort && s > 0) {
                    const long long t0 = clock64();
                    while (ld_acquire(&done[item.x]) < target) {
                        if (ld_relaxed(status) != 0) {
                            abort = 1;
                            break;
                        }
                        if (clock64() - t0 > wait_cycles) {
                            atomicCAS(status, 0, 1);
                            abort = 1;
                            break;
                        }
                        __nanosleep(100);
                    }
                }
                s_abort = abort;
            }
            __syncthreads();
            if (s_abort) return;
            const int par = (M.cur + s) & 1;
            if constexpr (HAS == HAS_MIXED && TY == 8) {
                if (M.storage == ST_F16) called_tile<__half, TY, HAS>(M, par, item.y, smem_raw);
                else if (M.storage == ST_BF16) called_tile<__nv_bfloat16, TY, HAS>(M, par, item.y, smem_raw);
                else called_tile<float, TY, HAS>(M, par, item.y, smem_raw);
            } else if (HAS == HAS_F16 || (HAS == HAS_MIXED && M.storage == ST_F16)) {
                ensemble_tile<__half, TY, HAS>(M, par, item.y, smem_raw);
            } else if (HAS == HAS_BF16 || (HAS == HAS_MIXED && M.storage == ST_BF16)) {
                ensemble_tile<__nv_bfloat16, TY, HAS>(M, par, item.y, smem_raw);
            } else {
                ensemble_tile<float, TY, HAS>(M, par, item.y, smem_raw);
            }
            __syncthreads();
            if (tid == 0) red_release_add(&done[item.x], 1u);
        }
    }
}

#define KIN_ENSEMBLE_PARAMS                                                                            \
    const EnsMember *__restrict__ mem, const int2 *__restrict__ items, int nitems, int nsteps, unsigned *done, \
        unsigned *next_item, int *status, long long wait_cycles, int stall_test

template <int TY, int HAS>
__global__ void __launch_bounds__(32 * block_warps(TY, HAS), blocks_an_sm(TY, HAS)) ensemble_kernel(KIN_ENSEMBLE_PARAMS) {
    ensemble_body<TY, HAS>(mem, items, nitems, nsteps, done, next_item, status, wait_cycles, stall_test);
}

// One LBE step of every member in tab[0 .. nmem) (one storage type): block b
// belongs to the member with the largest block0 <= b and takes blockDim.x * V
// consecutive cells of it (linear index x + N (y + N z)); each thread updates V
// cells of one row exactly as the standalone LBE step does.  FP32 blocks are
// held to 56 registers a thread, nine 128-thread blocks an SM (the 2-byte
// vector forms would spill there).
template <typename S>
__global__ void __launch_bounds__(128, sizeof(S) == 4 ? 9 : 1) lbe_batch_kernel(const LbeMember* __restrict__ tab, int nmem, int step) {
    const unsigned b = blockIdx.x;
    int lo = 0, hi = nmem - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (tab[mid].block0 <= b) lo = mid;
        else hi = mid - 1;
    }
    const LbeMember& M = tab[lo];
    const int N = M.N, V = M.V;
    // N <= 1024: cell indices fit in 32 bits
    const unsigned n3 = (unsigned)N * N * N, nn = (unsigned)N * N;
    const unsigned c = ((b - M.block0) * blockDim.x + threadIdx.x) * V;
    if (c >= n3) return;
    const size_t plane = n3;
    const int z = (int)(c / nn), r = (int)(c - z * nn), y = r / N, x = r - y * N;
    const int par = (M.cur + step) & 1;
    const S* src = static_cast<const S*>(M.buf[par]);
    S* dst = static_cast<S*>(M.buf[par ^ 1]);
    const MrtRates<float> rates = M.rates;
    if constexpr (sizeof(S) == 2) {
        if (V == 4) return lbe_vnode4p<S>(src, dst, N, plane, x, y, z, rates);
        if (V == 2) return lbe_vnode<S, 2>(src, dst, N, plane, x, y, z, rates);
    }
    lbe_node<S>(src, dst, N, plane, x, y, z, rates);
}

KIN_DEBUG_ACCESSOR(debug_word_ensemble)

}  // namespace kin

using namespace kin;

// Threads per block of the batched LBE launches when the caller has not chosen.
constexpr int kLbeBlock = 128;

struct kin_ensemble {
    std::vector<kin_sim*> members;
    std::vector<int> dugks_ids, lbe_ids;  // members of each scheme, in member order
    int has = 0;                          // the DUGKS members' storage types (HAS_*)
    int device = 0;
    cudaStream_t stream = nullptr;  // persistent DUGKS launch (and the graph's origin)
    cudaStream_t side = nullptr;    // batched LBE launches inside the graph
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    int tile_y = 5, lbe_block = kLbeBlock;
    int zchunk = 0;  // 0: chosen for the members (default_zchunk)
    int zc = 1;      // planes per item in use
    EnsMember* d_mem = nullptr;
    LbeMember* d_lbe = nullptr;
    int2* d_items = nullptr;
    unsigned* d_done = nullptr;
    int* d_status = nullptr;
    int nitems = 0;  // DUGKS items per step
    int grid = 0;    // blocks of the persistent launch
    // batched LBE launches, one per storage type (FP32, FP16, BF16): their
    // members' range in the LBE table and their blocks per step
    int lbe_off[3] = {0, 0, 0}, lbe_count[3] = {0, 0, 0};
    unsigned lbe_blocks[3] = {0, 0, 0};
    double wait_seconds = 10.0;
    // graph cache keyed by step count
    std::map<int, cudaGraphExec_t> graphs;
    int64_t launches = 0;
};

namespace {

// Steps per graph when there are LBE members (one kernel node each).
constexpr int kMaxGraphSteps = 256;

int ens_fail(int code, const char* what, cudaError_t e) {
    return set_error(code, "%s: %s", what, cudaGetErrorString(e));
}

#define ECK(call)                                                                      \
    do {                                                                               \
        cudaError_t e_ = (call);                                                       \
        if (e_ != cudaSuccess) return ens_fail(KIN_ECUDA, #call, e_);                  \
    } while (0)

void drop_graphs(kin_ensemble* e) {
    for (auto& kv : e->graphs) cudaGraphExecDestroy(kv.second);
    e->graphs.clear();
}

template <int TY, int HAS>
size_t persistent_smem() {
    const size_t fp32 = fused_smem_bytes<float, rows32(TY, HAS)>();
    return HAS == HAS_F32 ? fp32 : std::max(fp32, two_byte::tile_smem_bytes<__half, TY>());
}

template <int TY, int HAS>
int configure(kin_ensemble* e) {
    const size_t smem = persistent_smem<TY, HAS>();
    ECK(cudaFuncSetAttribute(ensemble_kernel<TY, HAS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem));
    int per_sm = 0, nsm = 0;
    ECK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, ensemble_kernel<TY, HAS>, 32 * block_warps(TY, HAS),
                                                      smem));
    ECK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, e->device));
    if (per_sm < 1) return set_error(KIN_ECUDA, "ensemble kernel does not fit on an SM");
    e->grid = std::min(per_sm * nsm, std::max(e->nitems, 1));
    return KIN_OK;
}

// f(tile height, storage types) of the kernel that this ensemble runs, as constants.
template <typename F>
auto with_kernel(const kin_ensemble* e, F&& f) {
    auto of_height = [&](auto ty) {
        switch (e->has) {
            case HAS_F32: return f(ty, std::integral_constant<int, HAS_F32>{});
            case HAS_F16: return f(ty, std::integral_constant<int, HAS_F16>{});
            case HAS_BF16: return f(ty, std::integral_constant<int, HAS_BF16>{});
        }
        return f(ty, std::integral_constant<int, HAS_MIXED>{});
    };
    switch (e->tile_y) {
        case 4: return of_height(std::integral_constant<int, 4>{});
        case 5: return of_height(std::integral_constant<int, 5>{});
        case 6: return of_height(std::integral_constant<int, 6>{});
    }
    return of_height(std::integral_constant<int, 8>{});
}

int storage_group(int storage) { return storage == ST_F16 ? 1 : storage == ST_BF16 ? 2 : 0; }

// Cells a thread of the batched LBE launch updates: as the standalone step.
int lbe_vector(const kin_sim* s) {
    if (s->storage == ST_F32) return 1;
    return s->N % 4 == 0 ? 4 : s->N % 2 == 0 ? 2 : 1;
}

// Rows of the tiles when the caller has not chosen.  FP32: 5, two 6-warp blocks an SM
// (0.347 ms a step for the DUGKS members of the reference mix, against 0.369 with 4
// rows, 0.362 with 6, 0.404 with 8).  One 2-byte type: 8, as stand-alone (the DUGKS and
// LBE members of half the reference mix in FP16: 575 us, 4 rows 765, 5 rows 760, 6 rows
// 695).  A mixture: 6, the most rows whose block takes 255 registers (2 FP32 and 2 FP16
// 96^3 members of each scheme: 376 us, 4 rows 457, 5 rows 422, 8 rows 557).
int default_tile_y(int has) { return has == HAS_F32 ? 5 : has == HAS_MIXED ? 6 : 8; }

// Rows of the tiles of a DUGKS member.
int tile_rows(const kin_ensemble* e, const kin_sim* s) {
    return s->storage == ST_F32 ? rows32(e->tile_y, e->has) : e->tile_y;
}

// DUGKS table from the members' current state (buffers, parity, nu, dt).
std::vector<EnsMember> dugks_table(const kin_ensemble* e) {
    std::vector<EnsMember> tab(e->dugks_ids.size());
    for (size_t d = 0; d < tab.size(); ++d) {
        const kin_sim* s = e->members[e->dugks_ids[d]];
        EnsMember& M = tab[d];
        M.buf[0] = s->buf[0];
        M.buf[1] = s->buf[1];
        M.N = s->N;
        M.storage = s->storage;
        M.cur = s->cur;
        M.coef = dugks_coef<float>(s->nu, s->dt);
        const int zc = std::min(e->zc, s->N);
        M.tiles_x = (s->N + 29) / 30;
        const int rows = tile_rows(e, s);
        M.tiles_y = (s->N + rows - 1) / rows;
        M.zchunk = zc;
        M.ntiles = M.tiles_x * M.tiles_y * ((s->N + zc - 1) / zc);
    }
    return tab;
}

// LBE table, grouped by storage type (FP32, FP16, BF16), each group's blocks
// numbered from 0; fills the group ranges of e.
std::vector<LbeMember> lbe_table(kin_ensemble* e) {
    std::vector<LbeMember> tab;
    for (int g = 0; g < 3; ++g) {
        e->lbe_off[g] = (int)tab.size();
        unsigned long long blocks = 0;
        for (int m : e->lbe_ids) {
            const kin_sim* s = e->members[m];
            if (storage_group(s->storage) != g) continue;
            LbeMember L;
            L.buf[0] = s->buf[0];
            L.buf[1] = s->buf[1];
            L.N = s->N;
            L.cur = s->cur;
            L.V = lbe_vector(s);
            L.block0 = (unsigned)blocks;
            L.rates = lbe_rates<float>(s->nu);
            const unsigned long long threads = (unsigned long long)s->N * s->N * s->N / L.V;
            blocks += (threads + e->lbe_block - 1) / e->lbe_block;
            tab.push_back(L);
        }
        e->lbe_count[g] = (int)tab.size() - e->lbe_off[g];
        e->lbe_blocks[g] = (unsigned)std::min<unsigned long long>(blocks, 0xffffffffull);
    }
    return tab;
}

int launch_persistent_config(kin_ensemble* e) {
    if (e->nitems == 0) {
        e->grid = 0;
        return KIN_OK;
    }
    return with_kernel(e, [&](auto ty, auto has) { return configure<ty(), has()>(e); });
}

// Planes per item when the caller has not chosen: a step takes about its items'
// planes (and 1.1 plane-times of prologue each) spread over the resident
// blocks, but no less than any member's own items take on all of them, round by
// round: that member's next step waits for the last.  Without the second bound a
// mix with one large member gets a nearly empty second round (us a step, one
// 96^3 and one 24^3 DUGKS member beside LBE: 24 planes 122, the 14 chosen now 89.5,
// the best of a sweep 82 with 32; one of 50^3: 3 planes 22.3, 4 16.4).  The reference
// mix gets whole columns, at most 128 planes (0.347 ms a step of its DUGKS members; 16
// planes: 0.388, 32: 0.358, 64: 0.347).
int default_zchunk(const kin_ensemble* e) {
    int nsm = 0, top = 1;
    if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, e->device) != cudaSuccess || nsm <= 0) nsm = 152;
    const double slots = (double)nsm * blocks_an_sm(e->tile_y, e->has);
    for (int m : e->dugks_ids) top = std::max(top, e->members[m]->N);
    int best = 1;
    double best_cost = -1.0;
    for (int zc = top; zc >= 1; --zc) {
        double sum = 0.0, longest = 0.0;
        for (int m : e->dugks_ids) {
            const int N = e->members[m]->N, c = std::min(zc, N), nz = (N + c - 1) / c;
            const int rows = tile_rows(e, e->members[m]);
            const double cols = (double)((N + 29) / 30) * ((N + rows - 1) / rows);
            sum += cols * (N + 1.1 * nz);
            longest = std::max(longest, std::ceil(cols * nz / slots) * (c + 1.1));
        }
        const double cost = std::max(sum / slots, longest);
        if (best_cost < 0.0 || cost < best_cost) {
            best_cost = cost;
            best = zc;
        }
    }
    return best;
}

// Work list for the current tuning; items of big members first so their long
// critical paths start early.
int build_tables(kin_ensemble* e) {
    e->zc = e->zchunk > 0 ? e->zchunk : default_zchunk(e);
    const std::vector<EnsMember> tab = dugks_table(e);
    std::vector<int> order(tab.size());
    for (size_t d = 0; d < order.size(); ++d) order[d] = (int)d;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return tab[a].N > tab[b].N; });
    std::vector<int2> items;
    for (int d : order)
        for (int t = 0; t < tab[d].ntiles; ++t) items.push_back(make_int2(d, t));
    if (e->d_items) cudaFree(e->d_items);
    e->d_items = nullptr;
    e->nitems = (int)items.size();
    ECK(cudaMalloc(&e->d_items, sizeof(int2) * std::max<size_t>(items.size(), 1)));
    if (!items.empty())
        ECK(cudaMemcpy(e->d_items, items.data(), sizeof(int2) * items.size(), cudaMemcpyHostToDevice));
    lbe_table(e);
    for (int g = 0; g < 3; ++g)
        if (e->lbe_blocks[g] > (unsigned)INT_MAX)
            return set_error(KIN_EINVAL, "the LBE members need more than 2^31 - 1 thread blocks a step");
    drop_graphs(e);
    return launch_persistent_config(e);
}

// The tables for a changed tuning.
int retuned(kin_ensemble* e) {
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(e->device);
    const int r = build_tables(e);
    cudaSetDevice(prev);
    return r;
}

long long wait_cycles(const kin_ensemble* e) {
    int khz = 0;
    cudaDeviceGetAttribute(&khz, cudaDevAttrClockRate, e->device);
    if (khz <= 0) khz = 2000000;
    return (long long)(e->wait_seconds * 1e3 * khz);
}

template <int TY, int HAS>
cudaError_t launch_persistent_t(kin_ensemble* e, int nsteps, int stall_test) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(e->grid);
    cfg.blockDim = dim3(32, block_warps(TY, HAS));
    cfg.dynamicSmemBytes = persistent_smem<TY, HAS>();
    cfg.stream = e->stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const int nd = (int)e->dugks_ids.size();
    return cudaLaunchKernelEx(&cfg, ensemble_kernel<TY, HAS>, (const EnsMember*)e->d_mem,
                              (const int2*)e->d_items, e->nitems, nsteps, e->d_done, e->d_done + nd, e->d_status,
                              wait_cycles(e), stall_test);
}

int launch_persistent(kin_ensemble* e, int nsteps, int stall_test) {
    const cudaError_t err = with_kernel(
        e, [&](auto ty, auto has) { return launch_persistent_t<ty(), has()>(e, nsteps, stall_test); });
    if (err != cudaSuccess) return ens_fail(KIN_ECUDA, "ensemble launch", err);
    return KIN_OK;
}

// Step `step` (counted from the start of the launch) of every LBE member.
int launch_lbe(kin_ensemble* e, int step, cudaStream_t stream) {
    for (int g = 0; g < 3; ++g) {
        if (e->lbe_count[g] == 0) continue;
        const LbeMember* tab = e->d_lbe + e->lbe_off[g];
        const dim3 grid(e->lbe_blocks[g]), block(e->lbe_block);
        if (g == 0) lbe_batch_kernel<float><<<grid, block, 0, stream>>>(tab, e->lbe_count[g], step);
        else if (g == 1) lbe_batch_kernel<__half><<<grid, block, 0, stream>>>(tab, e->lbe_count[g], step);
        else lbe_batch_kernel<__nv_bfloat16><<<grid, block, 0, stream>>>(tab, e->lbe_count[g], step);
        const cudaError_t err = cudaGetLastError();
        if (err != cudaSuccess) return ens_fail(KIN_ECUDA, "batched LBE launch", err);
    }
    return KIN_OK;
}

int sync_members(kin_ensemble* e) {
    for (kin_sim* s : e->members) ECK(cudaStreamSynchronize(s->stream));
    return KIN_OK;
}

int refresh_tables(kin_ensemble* e) {
    static_assert(sizeof(EnsMember) % 8 == 0 && sizeof(LbeMember) % 8 == 0, "table entries hold pointers");
    const std::vector<EnsMember> d = dugks_table(e);
    const std::vector<LbeMember> l = lbe_table(e);
    if (!d.empty())
        ECK(cudaMemcpyAsync(e->d_mem, d.data(), sizeof(EnsMember) * d.size(), cudaMemcpyHostToDevice, e->stream));
    if (!l.empty())
        ECK(cudaMemcpyAsync(e->d_lbe, l.data(), sizeof(LbeMember) * l.size(), cudaMemcpyHostToDevice, e->stream));
    // the copies read the host vectors: finish them before they go out of scope
    ECK(cudaStreamSynchronize(e->stream));
    return KIN_OK;
}

// Graph of nsteps steps: the persistent DUGKS launch on e->stream and, forked
// onto e->side, one batched LBE launch per step.
int capture(kin_ensemble* e, int nsteps, cudaGraphExec_t* out) {
    const int nd = (int)e->dugks_ids.size();
    const bool dugks = e->nitems > 0, lbe = !e->lbe_ids.empty();
    const bool fork = dugks && lbe;
    cudaGraph_t g = nullptr;
    ECK(cudaStreamBeginCapture(e->stream, cudaStreamCaptureModeThreadLocal));
    int rl = KIN_OK;
    cudaError_t ce = cudaSuccess;
    if (dugks) {
        ce = cudaMemsetAsync(e->d_done, 0, sizeof(unsigned) * (nd + 1), e->stream);
        if (ce == cudaSuccess) ce = cudaMemsetAsync(e->d_status, 0, sizeof(int), e->stream);
    }
    cudaStream_t lbe_stream = e->stream;
    if (fork && ce == cudaSuccess) {
        ce = cudaEventRecord(e->ev_fork, e->stream);
        if (ce == cudaSuccess) ce = cudaStreamWaitEvent(e->side, e->ev_fork, 0);
        lbe_stream = e->side;
    }
    if (ce != cudaSuccess) rl = ens_fail(KIN_ECUDA, "graph capture", ce);
    if (rl == KIN_OK && dugks) rl = launch_persistent(e, nsteps, 0);
    for (int s = 0; s < nsteps && rl == KIN_OK && lbe; ++s) rl = launch_lbe(e, s, lbe_stream);
    if (fork) {
        // join the side stream even after an error, so the capture can end
        cudaEventRecord(e->ev_join, e->side);
        cudaStreamWaitEvent(e->stream, e->ev_join, 0);
    }
    ce = cudaStreamEndCapture(e->stream, &g);
    if (rl != KIN_OK) {
        if (g) cudaGraphDestroy(g);
        return rl;
    }
    if (ce != cudaSuccess) return ens_fail(KIN_ECUDA, "graph capture", ce);
    ce = cudaGraphInstantiate(out, g, 0);
    cudaGraphDestroy(g);
    if (ce != cudaSuccess) return ens_fail(KIN_ECUDA, "graph instantiate", ce);
    return KIN_OK;
}

int run(kin_ensemble* e, int nsteps, int stall_test) {
    if (int r = sync_members(e)) return r;
    if (int r = refresh_tables(e)) return r;
    if (stall_test) {
        // the persistent launch alone, with a member barrier it cannot pass
        const int nd = (int)e->dugks_ids.size();
        ECK(cudaMemsetAsync(e->d_done, 0, sizeof(unsigned) * (nd + 1), e->stream));
        ECK(cudaMemsetAsync(e->d_status, 0, sizeof(int), e->stream));
        if (int r = launch_persistent(e, nsteps, 1)) return r;
    } else {
        auto it = e->graphs.find(nsteps);
        if (it == e->graphs.end()) {
            cudaGraphExec_t ex = nullptr;
            if (int r = capture(e, nsteps, &ex)) return r;
            it = e->graphs.emplace(nsteps, ex).first;
        }
        ECK(cudaGraphLaunch(it->second, e->stream));
    }
    int status = 0;
    if (e->nitems > 0) ECK(cudaMemcpyAsync(&status, e->d_status, sizeof(int), cudaMemcpyDeviceToHost, e->stream));
    ECK(cudaStreamSynchronize(e->stream));
    e->launches += 1;
    if (status != 0) {
        // items of several steps may have run: no member's state is known to
        // be a whole step, so every member refuses work until it is set again
        for (kin_sim* s : e->members) s->invalid = true;
        return set_error(KIN_ETIMEOUT, "ensemble member barrier timed out; the members' states are undefined");
    }
    for (kin_sim* s : e->members) {
        s->cur ^= (nsteps & 1);
        s->step += nsteps;
        s->epoch += 1;
    }
    return KIN_OK;
}

}  // namespace

extern "C" {

int kin_ensemble_create(kin_sim* const* members, int n, kin_ensemble** out) {
    if (!out || n <= 0 || !members) return set_error(KIN_EINVAL, "bad ensemble arguments");
    *out = nullptr;
    int dev = -1;
    for (int m = 0; m < n; ++m) {
        const kin_sim* s = members[m];
        if (!s) return set_error(KIN_EINVAL, "NULL member %d", m);
        if (s->storage == ST_F64)
            return set_error(KIN_EINVAL, "ensemble members use KIN_F32, KIN_F16 or KIN_BF16 storage");
        if (s->scheme == KIN_DUGKS && s->storage != ST_F32 && s->N % 2)
            return set_error(KIN_EINVAL, "member %d: a DUGKS member with 2-byte storage needs an even N", m);
        if (dev >= 0 && s->device != dev) return set_error(KIN_EINVAL, "members on different devices");
        dev = s->device;
        for (int k = 0; k < m; ++k)
            if (members[k] == s) return set_error(KIN_EINVAL, "member %d listed twice", m);
    }
    kin_ensemble* e = new kin_ensemble();
    e->members.assign(members, members + n);
    for (int m = 0; m < n; ++m) {
        if (members[m]->scheme == KIN_DUGKS) {
            e->dugks_ids.push_back(m);
            e->has |= members[m]->storage == ST_F16 ? HAS_F16 : members[m]->storage == ST_BF16 ? HAS_BF16 : HAS_F32;
        } else {
            e->lbe_ids.push_back(m);
        }
    }
    if (e->has & (e->has - 1)) e->has = HAS_MIXED;
    e->tile_y = default_tile_y(e->has);
    e->device = dev;
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(dev);
    auto bail = [&](int code) {
        kin_ensemble_destroy(e);
        cudaSetDevice(prev);
        return code;
    };
    cudaError_t c;
    if ((c = cudaStreamCreateWithFlags(&e->stream, cudaStreamNonBlocking)) != cudaSuccess)
        return bail(ens_fail(KIN_ECUDA, "stream", c));
    if ((c = cudaStreamCreateWithFlags(&e->side, cudaStreamNonBlocking)) != cudaSuccess)
        return bail(ens_fail(KIN_ECUDA, "stream", c));
    if ((c = cudaEventCreateWithFlags(&e->ev_fork, cudaEventDisableTiming)) != cudaSuccess ||
        (c = cudaEventCreateWithFlags(&e->ev_join, cudaEventDisableTiming)) != cudaSuccess)
        return bail(ens_fail(KIN_ECUDA, "event", c));
    if ((c = cudaMalloc(&e->d_mem, sizeof(EnsMember) * n)) != cudaSuccess) return bail(ens_fail(KIN_ENOMEM, "table", c));
    if ((c = cudaMalloc(&e->d_lbe, sizeof(LbeMember) * n)) != cudaSuccess) return bail(ens_fail(KIN_ENOMEM, "table", c));
    // one completion counter per DUGKS member, then the work counter
    if ((c = cudaMalloc(&e->d_done, sizeof(unsigned) * (n + 1))) != cudaSuccess)
        return bail(ens_fail(KIN_ENOMEM, "counters", c));
    if ((c = cudaMalloc(&e->d_status, sizeof(int))) != cudaSuccess) return bail(ens_fail(KIN_ENOMEM, "status", c));
    if (int r = build_tables(e)) return bail(r);
    cudaSetDevice(prev);
    *out = e;
    return KIN_OK;
}

int kin_ensemble_set_tuning(kin_ensemble* e, int tile_y, int zchunk, int lbe_block) {
    if (!e) return set_error(KIN_EINVAL, "NULL ensemble");
    if (tile_y > 0 && tile_y != 4 && tile_y != 6 && tile_y != 8)
        return set_error(KIN_EINVAL, "tile_y must be 4, 6 or 8");
    if (lbe_block > 0 && (lbe_block % 32 || lbe_block > 128))
        return set_error(KIN_EINVAL, "lbe_block must be a multiple of 32, at most 128");
    if (tile_y > 0) e->tile_y = tile_y;
    if (zchunk > 0) e->zchunk = zchunk;
    if (lbe_block > 0) e->lbe_block = lbe_block;
    return retuned(e);
}

int kin_ensemble_reset_tuning(kin_ensemble* e) {
    if (!e) return set_error(KIN_EINVAL, "NULL ensemble");
    e->tile_y = default_tile_y(e->has);
    e->zchunk = 0;
    e->lbe_block = kLbeBlock;
    return retuned(e);
}

int kin_ensemble_step(kin_ensemble* e, int nsteps) {
    if (!e) return set_error(KIN_EINVAL, "NULL ensemble");
    if (nsteps < 0) return set_error(KIN_EINVAL, "negative step count");
    if (nsteps == 0) return KIN_OK;
    for (const kin_sim* s : e->members)
        if (s->invalid) return set_error(KIN_ESTATE, "a member's state is undefined (set it again first)");
    nvtxRangePushA("kin_ensemble_step");
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(e->device);
    // the persistent kernel numbers (step, item) pairs and member progress in
    // 32 bits, and a graph holds one LBE launch per step: split the steps
    // into launches of at most max_steps
    unsigned long long max_steps =
        std::max<unsigned long long>(1, (0xffffffffull - (unsigned long long)e->grid) / std::max(e->nitems, 1));
    if (!e->lbe_ids.empty()) max_steps = std::min<unsigned long long>(max_steps, kMaxGraphSteps);
    int r = KIN_OK;
    for (long long left = nsteps; left > 0 && r == KIN_OK;) {
        const int n = (int)std::min<unsigned long long>((unsigned long long)left, max_steps);
        r = run(e, n, 0);
        left -= n;
    }
    cudaSetDevice(prev);
    nvtxRangePop();
    return r;
}

int kin_ensemble_test_timeout(kin_ensemble* e, double seconds) {
    if (!e || !(seconds > 0.0)) return set_error(KIN_EINVAL, "bad arguments");
    if (e->nitems == 0) return set_error(KIN_EINVAL, "no DUGKS member: the ensemble has no member barrier");
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(e->device);
    const double keep = e->wait_seconds;
    e->wait_seconds = seconds;
    const int r = run(e, 2, 1);
    e->wait_seconds = keep;
    cudaSetDevice(prev);
    return r;
}

int kin_ensemble_info(const kin_ensemble* e, int* nitems, int* grid, int64_t* launches) {
    if (!e) return set_error(KIN_EINVAL, "NULL ensemble");
    if (nitems) *nitems = e->nitems + (int)(e->lbe_blocks[0] + e->lbe_blocks[1] + e->lbe_blocks[2]);
    if (grid) *grid = e->grid;
    if (launches) *launches = e->launches;
    return KIN_OK;
}

void kin_ensemble_destroy(kin_ensemble* e) {
    if (!e) return;
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(e->device);
    if (e->stream) cudaStreamSynchronize(e->stream);
    if (e->side) cudaStreamSynchronize(e->side);
    drop_graphs(e);
    if (e->d_items) cudaFree(e->d_items);
    if (e->d_mem) cudaFree(e->d_mem);
    if (e->d_lbe) cudaFree(e->d_lbe);
    if (e->d_done) cudaFree(e->d_done);
    if (e->d_status) cudaFree(e->d_status);
    if (e->ev_fork) cudaEventDestroy(e->ev_fork);
    if (e->ev_join) cudaEventDestroy(e->ev_join);
    if (e->side) cudaStreamDestroy(e->side);
    if (e->stream) cudaStreamDestroy(e->stream);
    cudaSetDevice(prev);
    delete e;
}

}  // extern "C"
