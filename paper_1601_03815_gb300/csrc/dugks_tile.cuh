// Fused DUGKS step (Sec. II.A, Eqs. 9-20): one launch, one read and one write
// of f-tilde per cell.
//
// Each CTA owns a 30 x TY column of cells and marches along z through a chunk
// of planes.  Warps 0..TY-1 own one row each (lanes 0 and 31 are the x halo);
// warp TY serves both halo rows, 0 and TY + 1, which need about half of a row's
// work (f-bar-plus and one y record), so that the TY + 1 warps are evenly
// loaded.  A thread keeps its column's f-bar-plus of planes z and z + 1 in
// registers and prefetches f-tilde of the plane after them.
//
// Interface reconstruction splits exactly between the two cells of a face.
// With G_i^t(X) = fbp_i(X + e_t) - fbp_i(X - e_t) the Eq. 13/15/16 value at the
// face between L and R = L + e_a is
//   fbar_i = P_i^a(L) + M_i^a(R),
//   P_i^a = (1/2 + h xi_ia) X_i - (h/4) sum_{t != a} xi_it G_i^t,
//   M_i^a = (1/2 - h xi_ia) X_i - (h/4) sum_{t != a} xi_it G_i^t,
// where X = fbp at the cell; summed over i, the face moments (Eq. 17) split the
// same way through the moments of X and their tangential differences.  The
// moments of X follow from those of f-tilde (Eq. 19 conserves density and
// momentum and relaxes Pi), so a cell forms them once, and a neighbour's
// difference needs four of them instead of sums over its populations; of the
// populations only the diagonal pairs have a tangential direction.  A cell
// builds a "side record" per axis and sign (the 5 velocity pairs crossing the
// face plus density and momentum); a face (Eqs. 17, 7, 18, 10) needs one
// record from each neighbour: x neighbours exchange records by warp shuffles,
// y neighbours through shared memory, z neighbours are the same thread one
// plane apart.
//
// Updates lag one plane so the z face uses one cell view per plane.  Two block
// barriers per plane: one publishes f-bar-plus of plane z + 1 and the y records
// of plane z, the other the y-face values.
//
// Opposite populations (2p+1, 2p+2) travel as one pair (pair_math.cuh): both
// always undergo the same operation with a fixed coefficient pattern, so one
// packed FP32x2 instruction serves both.  Flux sums are kept sign-folded,
// Dhat_p = (D_{2p+1}, -D_{2p+2}), so a face adds the same signed value to
// both members.
//
// What bounds it, 128^3 FP32 (11-row tiles): the shared-memory and shuffle pipe,
// 58 % of its wavefront rate, and latency between the two barriers (FMA pipe
// 42 %, issue 47 %).  Against the form that staged f-tilde in shared memory
// and summed the moments of every difference: 96.3 -> 62.1 M warp instructions,
// 154 -> 117 us at 128^3, 0.961 -> 0.773 ms at 256^3 (2.65 -> 3.30 TB/s
// algorithmic).  The steps of that: moments from f-tilde and f-tilde kept in
// registers 0.961 -> 0.928; two 6-warp blocks on an SM, which drift apart so that
// one's exchange overlaps the other's arithmetic, instead of one of 10 warps
// -> 0.84; one base address per thread and the z loop unrolled by two (no
// register moves), one warp for both halo rows -> 0.797; the own y-face
// values kept in registers -> 0.773.  Not kept: mbarriers between neighbouring
// rows in place of the block barriers (1.10), 16 warps at 128 registers (1.09:
// spills go to L2, the shared memory leaves no L1).
#pragma once

#include <type_traits>

#include "dugks_face.cuh"
#include "kin_common.cuh"
#include "kin_debug.cuh"
#include "pair_math.cuh"

namespace kin {

// ------------------------------------------------------------------ pair tables
constexpr int NC = 5;  // velocity pairs crossing a face

// Component a of the velocity of pair p (that of population 2p+1).
__host__ __device__ constexpr int pe(int p, int a) {
    return a == 0 ? pair_x(p) : a == 1 ? pair_y(p) : pair_z(p);
}
// k-th pair (k = 0..4) whose velocity has a nonzero A component.
__host__ __device__ constexpr int cross_pair(int A, int k) {
    int n = 0;
    for (int p = 0; p < NPAIR; ++p)
        if (pe(p, A) != 0) {
            if (n == k) return p;
            ++n;
        }
    return -1;
}
// Position of pair p in the list of axis A, or -1.
__host__ __device__ constexpr int cross_index(int A, int p) {
    int n = 0;
    for (int q = 0; q < NPAIR; ++q)
        if (pe(q, A) != 0) {
            if (q == p) return n;
            ++n;
        }
    return -1;
}
// The other nonzero axis of diagonal pair p crossing A (-1 for an axis pair).
__host__ __device__ constexpr int tang_axis(int p, int A) {
    for (int t = 0; t < 3; ++t)
        if (t != A && pe(p, t) != 0) return t;
    return -1;
}

// e_p . (x, y, z); the first nonzero component of every e_p is +1.
template <int P, typename C>
__device__ __forceinline__ C pdot(C x, C y, C z) {
    constexpr int X = pair_x(P), Y = pair_y(P), Z = pair_z(P);
    if constexpr (X != 0) {
        static_assert(X == 1, "pair velocity convention");
        if constexpr (Y != 0) return Y > 0 ? x + y : x - y;
        else if constexpr (Z != 0) return Z > 0 ? x + z : x - z;
        else return x;
    } else if constexpr (Y != 0) {
        static_assert(Y == 1, "pair velocity convention");
        if constexpr (Z != 0) return Z > 0 ? y + z : y - z;
        else return y;
    } else {
        static_assert(Z == 1, "pair velocity convention");
        return z;
    }
}

// ------------------------------------------------------------------ shared memory
// Four values that one thread writes or reads together: two pairs.
template <typename C>
struct alignas(16) Quad {
    Pr<C> a, b;
};

constexpr int NXQ = 5;  // quads of a cell's exchange record
constexpr int NBQ = 5;  // quads of an update base (19 values)

// Quad (or pair) arrays, all indexed [..][row][lane] with the same row and lane
// strides, so that every access of a thread is one base address plus a constant.
//   XCH   [2 slots][5]: f-bar-plus of planes z and z + 1, what neighbours read of
//         it: the diagonal pairs (3, 4), (5, 6), (7, 8) and the moments that the
//         x and y differences need, (j_x, Pi_xx, Pi_xy, Pi_xz) and
//         (j_y, Pi_yx, Pi_yy, Pi_yz)
//   MY    [4]: y-face M records: pairs (0, 1), (2, 3), (4, moments 0-1), (moments 2-3, -)
//   FY    [3]: y-face values: pairs (0, 1), (2, 3), (4, -)
//   BASE  [2 slots][5]: f-tilde-plus of planes z - 1 and z (Eq. 20), each column's
//         own; rows 1..TY
template <typename C, int TY>
struct FusedSmem {
    static constexpr int ROW = 32 * (int)sizeof(Quad<C>);
    static constexpr int QX = (TY + 2) * ROW, QB = TY * ROW;
    static constexpr int PAD = (int)sizeof(Quad<C>);  // lane 0 of row 0 reads one quad to its left
    static constexpr int XCH = PAD, MY = XCH + 2 * NXQ * QX, FY = MY + 4 * QX, BASE = FY + 3 * QX - ROW,
                         BYTES = BASE + ROW + 2 * NBQ * QB;
};

// One quad or pair at shared-memory address a + OFF.  volatile: ordered with
// the barriers.
template <int OFF>
__device__ __forceinline__ void lds(unsigned a, Quad<float>& q) {
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4 + %5];"
                 : "=f"(q.a.x), "=f"(q.a.y), "=f"(q.b.x), "=f"(q.b.y)
                 : "r"(a), "n"(OFF) : "memory");
}
template <int OFF>
__device__ __forceinline__ void lds(unsigned a, float2& q) {
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2 + %3];" : "=f"(q.x), "=f"(q.y) : "r"(a), "n"(OFF) : "memory");
}
template <int OFF>
__device__ __forceinline__ void lds(unsigned a, double2& q) {
    asm volatile("ld.shared.v2.f64 {%0, %1}, [%2 + %3];" : "=d"(q.x), "=d"(q.y) : "r"(a), "n"(OFF) : "memory");
}
template <int OFF>
__device__ __forceinline__ void lds(unsigned a, Quad<double>& q) {
    lds<OFF>(a, q.a);
    lds<OFF + 16>(a, q.b);
}
template <int OFF>
__device__ __forceinline__ void sts(unsigned a, float2 p, float2 q) {
    asm volatile("st.shared.v4.f32 [%0 + %1], {%2, %3, %4, %5};" ::"r"(a), "n"(OFF), "f"(p.x), "f"(p.y), "f"(q.x), "f"(q.y) : "memory");
}
template <int OFF>
__device__ __forceinline__ void sts(unsigned a, float2 p) {
    asm volatile("st.shared.v2.f32 [%0 + %1], {%2, %3};" ::"r"(a), "n"(OFF), "f"(p.x), "f"(p.y) : "memory");
}
template <int OFF>
__device__ __forceinline__ void sts(unsigned a, double2 p) {
    asm volatile("st.shared.v2.f64 [%0 + %1], {%2, %3};" ::"r"(a), "n"(OFF), "d"(p.x), "d"(p.y) : "memory");
}
template <int OFF>
__device__ __forceinline__ void sts(unsigned a, double2 p, double2 q) {
    sts<OFF>(a, p);
    sts<OFF + 16>(a, q);
}

template <typename S, int TY>
constexpr size_t fused_smem_bytes() {
    return FusedSmem<typename Traits<S>::C, TY>::BYTES;
}

// ------------------------------------------------------------------ cells
// f-bar-plus of one cell with its moments.
template <typename C>
struct Cell {
    Pr<C> X[NPAIR];
    Pr<C> rj, jj;       // halves: (delta-rho, j_x) / 2, (j_y, j_z) / 2
    Quad<C> m[3];       // m[a] = (j_a, Pi_a0, Pi_a1, Pi_a2)
};

// Differences across a cell along one axis T: the two diagonal pairs named and
// (DJ_T, DP_0T, DP_1T, DP_2T).
template <typename C>
__device__ __forceinline__ Quad<C> qsub(const Quad<C>& p, const Quad<C>& m) {
    return Quad<C>{psub(p.a, m.a), psub(p.b, m.b)};
}
template <typename C>
__device__ __forceinline__ Quad<C> qadd(const Quad<C>& p, const Quad<C>& m) {
    return Quad<C>{padd(p.a, m.a), padd(p.b, m.b)};
}

// ------------------------------------------------------------------ side records
template <typename C>
struct Rec {
    Pr<C> r[NC];   // pairs crossing the face, in cross_pair order
    Pr<C> m0, m1;  // (density, momentum x), (momentum y, z)
};

// P (cell on the lower side of the face along A) and M (upper side) records.
// g[k], k = 1..4: the tangential difference of diagonal pair cross_pair(A, k);
// d: the sum of the moment differences along the two tangential axes.
template <int A, bool WANT_P, bool WANT_M, typename C>
__device__ __forceinline__ void side_records(const Cell<C>& v, const Pr<C> (&g)[NC], const Quad<C>& d,
                                             const DugksCoef<C>& k, Rec<C>& P, Rec<C>& M) {
    const Pr<C> b0 = pfma(k.mhq2, d.a, v.rj);
    const Pr<C> b1 = pfma(k.mhq2, d.b, v.jj);
    if constexpr (WANT_P) {
        P.m0 = pfma(k.h2, v.m[A].a, b0);
        P.m1 = pfma(k.h2, v.m[A].b, b1);
    }
    if constexpr (WANT_M) {
        M.m0 = pfma(k.mh2, v.m[A].a, b0);
        M.m1 = pfma(k.mh2, v.m[A].b, b1);
    }
    static_for<0, NC>([&](auto kc) {
        constexpr int K = decltype(kc)::value;
        constexpr int p = cross_pair(A, K);
        constexpr int sg = pe(p, A);
        // (1/2 + h xi_iA) for the two members: P uses cpp when e_pA = +1
        [[maybe_unused]] const Pr<C> cP = sg > 0 ? k.cpp : k.cpm;
        [[maybe_unused]] const Pr<C> cM = sg > 0 ? k.cpm : k.cpp;
        if constexpr (p < 3) {
            // the axis pair (K = 0): M carries fbp, the face scales it, so that no
            // product feeds a plain addition (which the compiler may contract in one
            // inlined copy and not in another)
            if constexpr (WANT_P) P.r[K] = pmul(cP, v.X[p]);
            if constexpr (WANT_M) M.r[K] = v.X[p];
        } else {
            constexpr int T = tang_axis(p, A);
            constexpr int tau = pe(p, T);
            // -(h/4) xi_iT G_i^T for both members
            const Pr<C> ht = pmul(tau > 0 ? k.hqp : k.hqm, g[K]);
            if constexpr (WANT_P) P.r[K] = pfma(cP, v.X[p], ht);
            if constexpr (WANT_M) M.r[K] = pfma(cM, v.X[p], ht);
        }
    });
}

// Face values f_i(x_b, t + h) = c1 fbar_i + c2 f_eq_i (Eqs. 17, 7, 18) of the
// pairs crossing the face along A, from the two side records.
template <int A, typename C>
__device__ __forceinline__ void face_values(const Rec<C>& P, const Rec<C>& M, const DugksCoef<C>& k,
                                            Pr<C> (&ff)[NC]) {
    const Pr<C> m0 = padd(P.m0, M.m0), m1 = padd(P.m1, M.m1);
    const C rho = m0.x, ux = m0.y, uy = m1.x, uz = m1.y;
    const C a0 = fma(C(-1.5), fma(uz, uz, fma(uy, uy, ux * ux)), rho);
    const C wa_ax = k.qw[0] * a0, wa_dg = k.qw[1] * a0;
    static_for<0, NC>([&](auto kc) {
        constexpr int K = decltype(kc)::value;
        constexpr int p = cross_pair(A, K);
        constexpr int cls = p < 3 ? 0 : 1;
        const C s = pdot<p>(ux, uy, uz);
        const C q = fma(k.qk[cls] * s, s, cls == 0 ? wa_ax : wa_dg);  // c2 W (a0 + 9/2 s^2)
        // +/- c2 3W s
        const Pr<C> fb = K == 0 ? pfma(k.cpm, M.r[K], P.r[K]) : padd(P.r[K], M.r[K]);
        ff[K] = pfma(k.c1p, fb, pmk(fma(k.ql[cls], s, q), fma(-k.ql[cls], s, q)));
    });
}

template <typename C>
__device__ __forceinline__ Pr<C> pshfl(Pr<C> v, int lane) {
    return pmk(__shfl_sync(0xffffffffu, v.x, lane), __shfl_sync(0xffffffffu, v.y, lane));
}
template <typename C>
__device__ __forceinline__ Pr<C> pshfl_down1(Pr<C> v) {
    return pmk(__shfl_down_sync(0xffffffffu, v.x, 1), __shfl_down_sync(0xffffffffu, v.y, 1));
}
template <typename C>
__device__ __forceinline__ Pr<C> pshfl_up1(Pr<C> v) {
    return pmk(__shfl_up_sync(0xffffffffu, v.x, 1), __shfl_up_sync(0xffffffffu, v.y, 1));
}

template <typename T>
__device__ __forceinline__ T opaque(T v) {
    asm volatile("" : "+r"(v));
    return v;
}
__device__ __forceinline__ int wrapc(int v, int n) {
    v %= n;
    return v < 0 ? v + n : v;
}

// ------------------------------------------------------------------ the tile
// One tile (tile coordinates bx, by, bz) of the fused step, run by a
// 32 x (TY + 1) thread block with fused_smem_bytes<S, TY>() of dynamic shared
// memory at smem_raw (16-byte aligned).  Also called by the persistent
// ensemble kernel.  With VEL (FP32-computed storage) the tile also writes
// rho0 u = sum xi f of the stored new state (Eq. 8) to uvel[3][N^3], summed in
// population order.  With WRAP (N <= 32) a warp holds whole periodic rows, lane
// = x, and needs no x halo: one tile along x where 31 and 32 cells take two.
template <typename S, int TY, bool VEL = false, bool WRAP = false>
__device__ __forceinline__ void dugks_tile(const S* __restrict__ src, S* __restrict__ dst, int N,
                                           int bx, int by, int bz, int zchunk,
                                           const DugksCoef<typename Traits<S>::C>& kc,
                                           unsigned char* smem_raw, float* __restrict__ uvel = nullptr) {
    using C = typename Traits<S>::C;
    using P2 = Pr<C>;
    using Q4 = Quad<C>;
    using SM = FusedSmem<C, TY>;
    static_assert(std::is_same<S, C>::value, "FP32 or FP64 storage (FP16 and BF16: dugks_tile16.cuh)");
    static_assert(!VEL || std::is_same<C, float>::value, "the fused velocity serves FP32-computed storage");

    // read once: recomputed from the special registers and the layout, the
    // shared-memory addresses cost ~20 instructions a plane
    const int lane = opaque((int)threadIdx.x);
    const bool halo = threadIdx.y == TY;
    const int row = opaque(halo ? 0 : (int)threadIdx.y + 1);
    // Every shared-memory access is own (or own + (TY + 1) rows in the halo warp) plus a
    // constant.  Of the arrays of TY + 2 rows that reaches one row up or down of rows 1
    // to TY and one quad beside a row; of the bases rows 1 to TY.
    static_assert(SM::XCH >= (int)sizeof(Q4) && SM::MY == SM::XCH + 2 * NXQ * SM::QX && SM::FY == SM::MY + 4 * SM::QX &&
                      SM::BASE + SM::ROW == SM::FY + 3 * SM::QX && SM::BYTES == SM::BASE + SM::ROW + 2 * NBQ * SM::QB,
                  "the arrays follow one another");
    (void)KIN_CHECK((int)threadIdx.y <= TY && lane < 32, DBG_DUGKS_ROW, threadIdx.y);
    (void)KIN_CHECK(row >= 0 && row <= TY && (halo ? row == 0 : row >= 1), DBG_DUGKS_SLOT, row);
    const unsigned own = opaque((unsigned)__cvta_generic_to_shared(smem_raw) + row * SM::ROW + lane * (int)sizeof(Q4));
    const int z0 = bz * zchunk;
    const int zend = min(z0 + zchunk, N);
    const int gxr = WRAP ? lane : bx * 30 - 1 + lane, gyr = by * TY - 1 + row;
    const int gx = wrapc(gxr, N), gy = wrapc(gyr, N);
    const bool valid = (WRAP || (lane >= 1 && lane <= 30)) && gxr < N && gyr < N;
    // WRAP: the lanes of the x neighbours and their distance in shared memory
    [[maybe_unused]] const int right = WRAP ? (lane + 1 == N ? 0 : min(lane + 1, 31)) : 0;
    [[maybe_unused]] const int left = WRAP ? (lane == 0 ? N - 1 : lane - 1) : 0;
    (void)KIN_CHECK(right >= 0 && right < 32 && left >= 0 && left < 32, DBG_DUGKS_SLOT, right * 64 + left);
    [[maybe_unused]] const int to_right = (right - lane) * (int)sizeof(Q4), to_left = (left - lane) * (int)sizeof(Q4);
    const size_t plane = (size_t)N * N * N;
    // cell indices fit in 32 bits (N <= 1024)
    const unsigned nn32 = (unsigned)N * N, col32 = (unsigned)gx + (unsigned)N * gy;

    auto zwrap = [&](int z) { return z < 0 ? z + N : (z >= N ? z - N : z); };

    // f-tilde of a column at plane z, from L2 (kin_launch.cuh; in the persistent
    // ensemble kernel other blocks wrote it earlier in the same launch)
    auto load_plane = [&](int z, unsigned col, C (&fr)[Q]) {
        const unsigned o = (unsigned)zwrap(z) * nn32 + col;
        if (!KIN_CHECK(o < plane, DBG_DUGKS_LOAD, o)) return;
#pragma unroll
        for (int i = 0; i < Q; ++i) fr[i] = Traits<S>::load_l2(src + i * plane + o);
    };

    // Eq. 19 of the column's values: fbp = f + b (f_eq - f), f_eq of a pair
    // = q +/- l (Eq. 7), with the moments of fbp: delta-rho and j are those of
    // f, Pi = Pi_f + b (Pi_eq - Pi_f) with Pi_eq = delta-rho / 3 I + j j.  The
    // exchange record goes to slot SL.  With KEEP also f-tilde-plus = 4/3 fbp -
    // 1/3 f-tilde (Eq. 20), kept in the column's own slot until the update.
    auto prestep = [&](auto slc, auto keepc, unsigned own, const C (&fr)[Q], Cell<C>& n) {
        constexpr int SL = decltype(slc)::value;
        constexpr bool keep = decltype(keepc)::value;
        P2 f[NPAIR];
#pragma unroll
        for (int q = 0; q < NPAIR; ++q) f[q] = pmk(fr[2 * q + 1], fr[2 * q + 2]);
        const C f0 = fr[0];
        C a[NPAIR], b[NPAIR];
#pragma unroll
        for (int q = 0; q < NPAIR; ++q) {
            a[q] = f[q].x + f[q].y;
            b[q] = f[q].x - f[q].y;
        }
        const C s34 = a[3] + a[4], s56 = a[5] + a[6], s78 = a[7] + a[8];
        const C drho = f0 + (((a[0] + a[1]) + a[2]) + ((s34 + s56) + s78));
        const C jx = (b[0] + b[3]) + (b[4] + (b[5] + b[6]));
        const C jy = (b[1] + b[3]) - (b[4] - (b[7] + b[8]));
        const C jz = (b[2] + b[5]) - (b[6] - (b[7] - b[8]));
        const C r3 = mul_rn(drho, C(1) / C(3));
        auto relax = [&](C pf, C ja, C jb, C r) { return fma(kc.b, fma(ja, jb, r - pf), pf); };
        const C pxx = relax(a[0] + (s34 + s56), jx, jx, r3);
        const C pyy = relax(a[1] + (s34 + s78), jy, jy, r3);
        const C pzz = relax(a[2] + (s56 + s78), jz, jz, r3);
        const C pxy = relax(a[3] - a[4], jx, jy, C(0));
        const C pxz = relax(a[5] - a[6], jx, jz, C(0));
        const C pyz = relax(a[7] - a[8], jy, jz, C(0));
        n.rj = pmk(C(0.5) * drho, C(0.5) * jx);
        n.jj = pmk(C(0.5) * jy, C(0.5) * jz);
        n.m[0] = Q4{pmk(jx, pxx), pmk(pxy, pxz)};
        n.m[1] = Q4{pmk(jy, pxy), pmk(pyy, pyz)};
        n.m[2] = Q4{pmk(jz, pxz), pmk(pyz, pzz)};
        constexpr int X = SM::XCH + SL * NXQ * SM::QX;
        constexpr int B = SM::BASE + SL * NBQ * SM::QB;
        sts<X + 3 * SM::QX>(own, n.m[0].a, n.m[0].b);
        sts<X + 4 * SM::QX>(own, n.m[1].a, n.m[1].b);
        const C a0 = fma(C(-1.5), fma(jz, jz, fma(jy, jy, jx * jx)), drho);
        const C wa_ax = (C(2) / C(36)) * a0, wa_dg = (C(1) / C(36)) * a0;
        P2 t[NPAIR];
        static_for<0, NPAIR>([&](auto pc) {
            constexpr int PP = decltype(pc)::value;
            constexpr bool AX = PP < 3;
            const C sd = pdot<PP>(jx, jy, jz);
            // W (a0 + 9/2 s^2) with 9/2 W = 1/4 (axis) or 1/8 (diagonal)
            const C q = fma(C(AX ? 0.25 : 0.125) * sd, sd, AX ? wa_ax : wa_dg);
            constexpr C w3 = lin3w<C>(AX ? 1 : 2);
            n.X[PP] = pfma(kc.b2, psub(pmk(fma(w3, sd, q), fma(-w3, sd, q)), f[PP]), f[PP]);
            t[PP] = pfma(kc.third, psub(n.X[PP], f[PP]), n.X[PP]);
            if constexpr (PP == 4) sts<X>(own, n.X[3], n.X[4]);
            if constexpr (PP == 6) sts<X + SM::QX>(own, n.X[5], n.X[6]);
            if constexpr (PP == 8) sts<X + 2 * SM::QX>(own, n.X[7], n.X[8]);
            if constexpr (PP % 2 == 1) {
                if constexpr (keep) sts<B + (PP / 2) * SM::QB>(own, t[PP - 1], t[PP]);
            }
        });
        if constexpr (keep) {
            const C X0 = fma(kc.b, fma(C(12) / C(36), a0, -f0), f0);
            sts<B + 4 * SM::QB>(own, t[8], pmk(fma(C(1.0 / 3.0), X0 - f0, X0), C(0)));
        }
    };

    // differences of quad K of exchange slot SL along x and y.  The outer lanes
    // read past their row: their x differences are never used.
    auto diff_x = [&](auto slc, auto kc2, unsigned own) {
        constexpr int O = SM::XCH + decltype(slc)::value * NXQ * SM::QX + decltype(kc2)::value * SM::QX;
        Q4 p, m;
        if constexpr (WRAP) {
            lds<O>(own + to_right, p);
            lds<O>(own + to_left, m);
        } else {
            lds<O + (int)sizeof(Q4)>(own, p);
            lds<O - (int)sizeof(Q4)>(own, m);
        }
        return qsub<C>(p, m);
    };
    auto diff_y = [&](auto slc, auto kc2) {
        constexpr int O = SM::XCH + decltype(slc)::value * NXQ * SM::QX + decltype(kc2)::value * SM::QX;
        Q4 p, m;
        lds<O + SM::ROW>(own, p);
        lds<O - SM::ROW>(own, m);
        return qsub<C>(p, m);
    };
    constexpr auto k0 = std::integral_constant<int, 0>{};
    constexpr auto k1 = std::integral_constant<int, 1>{};
    constexpr auto k2 = std::integral_constant<int, 2>{};
    constexpr auto k3 = std::integral_constant<int, 3>{};
    constexpr auto k4 = std::integral_constant<int, 4>{};

    auto y_face = [&](const Rec<C>& Py, unsigned own, P2 (&ffy)[NC]) {
        // face between this row and the one above
        Rec<C> Mu;
        Q4 q0, q1, q2;
        lds<SM::MY + SM::ROW>(own, q0);
        lds<SM::MY + SM::QX + SM::ROW>(own, q1);
        lds<SM::MY + 2 * SM::QX + SM::ROW>(own, q2);
        lds<SM::MY + 3 * SM::QX + SM::ROW>(own, Mu.m1);
        Mu.r[0] = q0.a, Mu.r[1] = q0.b, Mu.r[2] = q1.a, Mu.r[3] = q1.b, Mu.r[4] = q2.a;
        Mu.m0 = q2.b;
        face_values<1>(Py, Mu, kc, ffy);
        sts<SM::FY>(own, ffy[0], ffy[1]);
        sts<SM::FY + SM::QX>(own, ffy[2], ffy[3]);
        sts<SM::FY + 2 * SM::QX>(own, ffy[4]);
    };
    auto sync = [] { asm volatile("bar.sync 0, %0;" ::"n"(32 * (TY + 1)) : "memory"); };

    if (halo) {
        // rows 0 and TY + 1: f-bar-plus for their neighbours, the P record of row
        // 0 with its y face, the M record of row TY + 1
        const unsigned ownr[2] = {own, own + (TY + 1) * SM::ROW};
        const unsigned col[2] = {col32, (unsigned)gx + (unsigned)N * wrapc(by * TY + TY, N)};
        Cell<C> A[2], B[2];
        C fr[2][Q];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            load_plane(z0 - 1, col[r], fr[r]);
            prestep(k1, std::false_type{}, ownr[r], fr[r], B[r]);
            load_plane(z0, col[r], fr[r]);
            prestep(k0, std::false_type{}, ownr[r], fr[r], A[r]);
            if (z0 + 1 <= zend) load_plane(z0 + 1, col[r], fr[r]);
        }
        sync();
        auto advance = [&](auto slc, int z, Cell<C> (&cur)[2], Cell<C> (&nxt)[2]) -> bool {
            constexpr auto other = std::integral_constant<int, decltype(slc)::value ^ 1>{};
            sync();
            if (z == zend) return true;
            Rec<C> Py, My, unused;
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const Q4 zp78{nxt[r].X[7], nxt[r].X[8]}, zpm = nxt[r].m[2];
                prestep(other, std::false_type{}, ownr[r], fr[r], nxt[r]);
                const Q4 z78 = qsub<C>(Q4{nxt[r].X[7], nxt[r].X[8]}, zp78), zm = qsub<C>(nxt[r].m[2], zpm);
                if (z + 2 <= zend) load_plane(z + 2, col[r], fr[r]);
                const Q4 xp = diff_x(slc, k0, ownr[r]), xm = diff_x(slc, k3, ownr[r]);
                const P2 g[NC] = {P2{}, xp.a, xp.b, z78.a, z78.b};
                if (r == 0) {
                    side_records<1, true, false>(cur[r], g, qadd<C>(xm, zm), kc, Py, unused);
                } else {
                    side_records<1, false, true>(cur[r], g, qadd<C>(xm, zm), kc, unused, My);
                    sts<SM::MY>(ownr[r], My.r[0], My.r[1]);
                    sts<SM::MY + SM::QX>(ownr[r], My.r[2], My.r[3]);
                    sts<SM::MY + 2 * SM::QX>(ownr[r], My.r[4], My.m0);
                    sts<SM::MY + 3 * SM::QX>(ownr[r], My.m1);
                }
            }
            sync();
            P2 ffy[NC];
            y_face(Py, ownr[0], ffy);
            return false;
        };
        for (int z = z0;; z += 2) {
            if (advance(k0, z, A, B)) return;
            if (advance(k1, z + 1, B, A)) return;
        }
    }

    Cell<C> A, B;          // planes z and z - 1, in turn
    C fr[Q];
    Rec<C> Pz;             // P^z record of plane z - 1
    P2 ffy[NC] = {};       // upper y-face values of plane z - 1
    P2 D[NPAIR];           // sign-folded flux sums of plane z - 1, still missing z and y faces
#pragma unroll
    for (int q = 0; q < NPAIR; ++q) D[q] = pmk(C(0), C(0));

    // prologue: planes z0 - 1 (slot 1) and z0 (slot 0)
    load_plane(z0 - 1, col32, fr);
    prestep(k1, std::false_type{}, own, fr, B);
    load_plane(z0, col32, fr);
    prestep(k0, std::true_type{}, own, fr, A);
    if (z0 + 1 <= zend) load_plane(z0 + 1, col32, fr);
    sync();
    {
        const Q4 xq = diff_x(k1, k1, own), xm = diff_x(k1, k3, own), yq = diff_y(k1, k2), ym = diff_y(k1, k4);
        const P2 g[NC] = {P2{}, xq.a, xq.b, yq.a, yq.b};
        Rec<C> unused;
        side_records<2, true, false>(B, g, qadd<C>(xm, ym), kc, Pz, unused);
    }

    // One plane: cur is plane z (exchange slot SL), nxt holds plane z - 1 and
    // leaves with plane z + 1.
    auto advance = [&](auto slc, int z, Cell<C>& cur, Cell<C>& nxt) -> bool {
        constexpr int SL = decltype(slc)::value;
        constexpr auto other = std::integral_constant<int, SL ^ 1>{};
        const bool last = z == zend;
        const Q4 xm = diff_x(slc, k3, own), ym = diff_y(slc, k4);
        P2 ffz[NC];
        {
            // z face (z - 1, z): P^z(z - 1) carried, M^z(z) from this plane
            const Q4 xq = diff_x(slc, k1, own), yq = diff_y(slc, k2);
            Rec<C> Pn, Mz;
            const P2 g[NC] = {P2{}, xq.a, xq.b, yq.a, yq.b};
            side_records<2, true, true>(cur, g, qadd<C>(xm, ym), kc, Pn, Mz);
            face_values<2>(Pz, Mz, kc, ffz);
            Pz = Pn;
            static_for<0, NC>([&](auto kc2) {
                constexpr int K = decltype(kc2)::value;
                constexpr int p = cross_pair(2, K);
                D[p] = padd_sg<pe(p, 2)>(D[p], ffz[K]);
            });
        }
        sync();  // fy of plane z - 1 complete; slot SL ^ 1 (plane z - 1) no longer read
        // update plane z - 1 (Eqs. 20, 9)
        if (z > z0) {
            Q4 l0, l1;
            P2 l4;
            lds<SM::FY - SM::ROW>(own, l0);
            lds<SM::FY + SM::QX - SM::ROW>(own, l1);
            lds<SM::FY + 2 * SM::QX - SM::ROW>(own, l4);
            const P2 fl[NC] = {l0.a, l0.b, l1.a, l1.b, l4};
            static_for<0, NC>([&](auto kc2) {
                constexpr int K = decltype(kc2)::value;
                constexpr int p = cross_pair(1, K);
                constexpr int sg = pe(p, 1);
                const P2 d = psub(ffy[K], fl[K]);
                if constexpr (pe(p, 0) != 0 || pe(p, 2) != 0) {
                    D[p] = padd_sg<sg>(D[p], d);
                } else {
                    D[p] = sg > 0 ? d : pneg(d);
                }
            });
            P2 t[NPAIR + 1];
            static_for<0, NBQ>([&](auto qc) {
                constexpr int K = decltype(qc)::value;
                Q4 v;
                lds<SM::BASE + (SL ^ 1) * NBQ * SM::QB + K * SM::QB>(own, v);
                t[2 * K] = v.a;
                t[2 * K + 1] = v.b;
            });
            const unsigned c = (unsigned)(z - 1) * nn32 + col32;
            if (valid && KIN_CHECK(c < plane, DBG_DUGKS_STORE, c)) {
                [[maybe_unused]] C uv[3] = {C(0), C(0), C(0)};
                // velocity sums in population order: the same additions as the
                // separate velocity pass over the stored state
                [[maybe_unused]] auto vel_add = [&](auto ic, C v) {
                    constexpr int I = decltype(ic)::value;
                    if constexpr (cx(I) > 0) uv[0] += v;
                    if constexpr (cx(I) < 0) uv[0] -= v;
                    if constexpr (cy(I) > 0) uv[1] += v;
                    if constexpr (cy(I) < 0) uv[1] -= v;
                    if constexpr (cz(I) > 0) uv[2] += v;
                    if constexpr (cz(I) < 0) uv[2] -= v;
                };
                Traits<S>::store(dst + c, t[NPAIR].x);
                static_for<0, NPAIR>([&](auto pc) {
                    constexpr int PP = decltype(pc)::value;
                    // f-tilde-plus minus dt times the flux sum (Eq. 9)
                    const P2 r = pfma(kc.dts, D[PP], t[PP]);
                    __stcg(dst + (2 * PP + 1) * plane + c, r.x);
                    __stcg(dst + (2 * PP + 2) * plane + c, r.y);
                    if constexpr (VEL) {
                        vel_add(std::integral_constant<int, 2 * PP + 1>{}, r.x);
                        vel_add(std::integral_constant<int, 2 * PP + 2>{}, r.y);
                    }
                });
                if constexpr (VEL) {
                    uvel[c] = uv[0];
                    uvel[plane + c] = uv[1];
                    uvel[2 * plane + c] = uv[2];
                }
            }
        }
        if (last) return true;
        // plane z + 1
        const Q4 zp56{nxt.X[5], nxt.X[6]}, zp78{nxt.X[7], nxt.X[8]}, zpm = nxt.m[2];
        prestep(other, std::true_type{}, own, fr, nxt);
        const Q4 z56 = qsub<C>(Q4{nxt.X[5], nxt.X[6]}, zp56), z78 = qsub<C>(Q4{nxt.X[7], nxt.X[8]}, zp78);
        const Q4 zm = qsub<C>(nxt.m[2], zpm);
        {
            // x faces: this lane's face to the right uses the next lane's M record
            Rec<C> Px, Mx, Mn;
            const Q4 yp = diff_y(slc, k0);
            const P2 g[NC] = {P2{}, yp.a, yp.b, z56.a, z56.b};
            side_records<0, true, true>(cur, g, qadd<C>(ym, zm), kc, Px, Mx);
            auto from_right = [&](P2 v) { return WRAP ? pshfl<C>(v, right) : pshfl_down1<C>(v); };
#pragma unroll
            for (int k = 0; k < NC; ++k) Mn.r[k] = from_right(Mx.r[k]);
            Mn.m0 = from_right(Mx.m0);
            Mn.m1 = from_right(Mx.m1);
            P2 ffx[NC];
            face_values<0>(Px, Mn, kc, ffx);
            static_for<0, NC>([&](auto kc2) {
                constexpr int K = decltype(kc2)::value;
                constexpr int p = cross_pair(0, K);
                const P2 fl = WRAP ? pshfl<C>(ffx[K], left) : pshfl_up1<C>(ffx[K]);
                // Dhat = e_px (F(x + 1/2) - F(x - 1/2)), the first contribution
                D[p] = pe(p, 0) > 0 ? psub(ffx[K], fl) : psub(fl, ffx[K]);
            });
            static_for<0, NC>([&](auto kc2) {
                constexpr int K = decltype(kc2)::value;
                constexpr int p = cross_pair(2, K);
                constexpr int sg = pe(p, 2);
                if constexpr (pe(p, 0) != 0) D[p] = padd_sg<-sg>(D[p], ffz[K]);
                else D[p] = sg > 0 ? pneg(ffz[K]) : ffz[K];
            });
        }
        if (z + 2 <= zend) load_plane(z + 2, col32, fr);
        Rec<C> Py;
        {
            Rec<C> My;
            const Q4 xp = diff_x(slc, k0, own);
            const P2 g[NC] = {P2{}, xp.a, xp.b, z78.a, z78.b};
            side_records<1, true, true>(cur, g, qadd<C>(xm, zm), kc, Py, My);
            sts<SM::MY>(own, My.r[0], My.r[1]);
            sts<SM::MY + SM::QX>(own, My.r[2], My.r[3]);
            sts<SM::MY + 2 * SM::QX>(own, My.r[4], My.m0);
            sts<SM::MY + 3 * SM::QX>(own, My.m1);
        }
        sync();  // my of plane z and slot SL ^ 1 (plane z + 1) complete; fy of plane z - 1 consumed
        y_face(Py, own, ffy);
        return false;
    };
    for (int z = z0;; z += 2) {
        if (advance(k0, z, A, B)) break;
        if (advance(k1, z + 1, B, A)) break;
    }
}

// Coefficients of Eqs. 18-19 for viscosity nu (tau = nu / RT) and step dt,
// with the derived constants of the fused tile.
template <typename C>
inline DugksCoef<C> dugks_coef(double nu, double dt) {
    const double tau = 3.0 * nu, h = 0.5 * dt;
    DugksCoef<C> k{};
    k.a = C((2.0 * tau - h) / (2.0 * tau + dt));
    k.b = C(3.0 * h / (2.0 * tau + dt));
    k.h = C(h);
    k.c1 = C(2.0 * tau / (2.0 * tau + h));
    k.c2 = C(h / (2.0 * tau + h));
    k.dt = C(dt);
    k.hq = C(0.25 * h);
    const C c2 = k.c2;
    k.qk[0] = c2 * C(0.25);
    k.qk[1] = c2 * C(0.125);
    k.qw[0] = c2 * (C(2) / C(36));
    k.qw[1] = c2 * (C(1) / C(36));
    k.ql[0] = c2 * lin3w<C>(1);
    k.ql[1] = c2 * lin3w<C>(2);
    k.cpp = pmk(C(0.5 + h), C(0.5 - h));
    k.cpm = pmk(C(0.5 - h), C(0.5 + h));
    k.hqp = pmk(-k.hq, k.hq);
    k.hqm = pmk(k.hq, -k.hq);
    k.b2 = pmk(k.b, k.b);
    const C c1 = C(1) - c2;
    k.c1p = pmk(c1, c1);
    k.third = pmk(C(1.0 / 3.0), C(1.0 / 3.0));
    k.dts = pmk(-k.dt, k.dt);
    k.h2 = pmk(k.h, k.h);
    k.mh2 = pmk(-k.h, -k.h);
    k.mhq2 = pmk(-k.hq, -k.hq);
    return k;
}

}  // namespace kin
