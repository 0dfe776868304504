// Device-side lattice definitions shared by the libkin kernels.
//
// D3Q19 (Sec. II.A, Eq. 5): population 0 is at rest, 1..6 move along the axes,
// 7..18 along the face diagonals; opposite velocities occupy slots (2p+1, 2p+2)
// for p = 0..8.  This order is part of the library's public layout (kin.h).
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>
#include <utility>

namespace kin {

constexpr int Q = 19;
constexpr int NPAIR = 9;

// Velocity of the "positive" member of pair p (population 2p+1); the partner
// 2p+2 moves the opposite way.
__host__ __device__ constexpr int pair_x(int p) {
    return p == 0 ? 1 : p == 1 ? 0 : p == 2 ? 0 : p == 3 ? 1 : p == 4 ? 1 : p == 5 ? 1 : p == 6 ? 1 : 0;
}
__host__ __device__ constexpr int pair_y(int p) {
    return p == 0 ? 0 : p == 1 ? 1 : p == 2 ? 0 : p == 3 ? 1 : p == 4 ? -1 : p == 5 ? 0 : p == 6 ? 0 : 1;
}
__host__ __device__ constexpr int pair_z(int p) {
    return p == 0 ? 0 : p == 1 ? 0 : p == 2 ? 1 : p == 3 ? 0 : p == 4 ? 0 : p == 5 ? 1 : p == 6 ? -1
         : p == 7 ? 1 : -1;
}

// Velocity component a (0 = x, 1 = y, 2 = z) of population i.
__host__ __device__ constexpr int cx(int i) { return i == 0 ? 0 : ((i & 1) ? pair_x((i - 1) / 2) : -pair_x((i - 1) / 2)); }
__host__ __device__ constexpr int cy(int i) { return i == 0 ? 0 : ((i & 1) ? pair_y((i - 1) / 2) : -pair_y((i - 1) / 2)); }
__host__ __device__ constexpr int cz(int i) { return i == 0 ? 0 : ((i & 1) ? pair_z((i - 1) / 2) : -pair_z((i - 1) / 2)); }
__host__ __device__ constexpr int cc(int i, int a) { return a == 0 ? cx(i) : a == 1 ? cy(i) : cz(i); }

// Weights W_i (Sec. II.A) as exact rationals 12/36, 2/36, 1/36.
__host__ __device__ constexpr int w36(int i) { return i == 0 ? 12 : (i <= 6 ? 2 : 1); }

// ---------------------------------------------------------------------------
// a * b, never contracted with a following addition (code that is inlined in
// several places has to round the same way in each).
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// ---------------------------------------------------------------------------
// Compile-time loop: calls f(std::integral_constant<int, I>) for I in [B, E).
template <int B, int E, typename F>
__device__ __forceinline__ void static_for(F&& f) {
    if constexpr (B < E) {
        f(std::integral_constant<int, B>{});
        static_for<B + 1, E>(static_cast<F&&>(f));
    }
}

// ---------------------------------------------------------------------------
// Storage types.  Arithmetic runs in Traits<S>::C.
template <typename S>
struct Traits;
template <>
struct Traits<float> {
    using C = float;
    static __device__ __forceinline__ C load(const float* p) { return __ldg(p); }
    static __device__ __forceinline__ C load_l2(const float* p) { return __ldcg(p); }
    static __device__ __forceinline__ void store(float* p, C v) { *p = v; }
};
template <>
struct Traits<double> {
    using C = double;
    static __device__ __forceinline__ C load(const double* p) { return __ldg(p); }
    static __device__ __forceinline__ C load_l2(const double* p) { return __ldcg(p); }
    static __device__ __forceinline__ void store(double* p, C v) { *p = v; }
};
template <>
struct Traits<__half> {
    using C = float;
    static __device__ __forceinline__ C load(const __half* p) { return __half2float(__ldg(p)); }
    static __device__ __forceinline__ C load_l2(const __half* p) {
        return __half2float(__ushort_as_half(__ldcg(reinterpret_cast<const unsigned short*>(p))));
    }
    static __device__ __forceinline__ void store(__half* p, C v) { *p = __float2half_rn(v); }
};
template <>
struct Traits<__nv_bfloat16> {
    using C = float;
    static __device__ __forceinline__ C load(const __nv_bfloat16* p) {
        return __bfloat162float(__ldg(p));
    }
    static __device__ __forceinline__ C load_l2(const __nv_bfloat16* p) {
        return __bfloat162float(__ushort_as_bfloat16(__ldcg(reinterpret_cast<const unsigned short*>(p))));
    }
    static __device__ __forceinline__ void store(__nv_bfloat16* p, C v) { *p = __float2bfloat16_rn(v); }
};

// ---------------------------------------------------------------------------
// Coefficient 3 W_i of the linear term of Eq. 7 for |xi_i|^2 = r2 (1 or 2).
// Exactly, 2 (3 W_1) + 8 (3 W_7) = 1 makes sum_i xi_i f_eq_i = rho0 u.  In FP32
// the rounded values fl(1/6), fl(1/12) sum to 1 + 3e-8, which a DUGKS step
// multiplies into the momentum every step (f-bar-plus = f + b (f_eq - f));
// so FP32 uses fl(1/12) and the FP32 value 5592405 * 2^-25 for which the sum
// is exactly 1.  FP64 keeps 1/6 and 1/12.
template <typename C>
__host__ __device__ constexpr C lin3w(int r2) {
    if constexpr (sizeof(C) == 4) return r2 == 1 ? C(5592405.0 / 33554432.0) : C(11184811.0 / 134217728.0);
    else return r2 == 1 ? C(1.0 / 6.0) : C(1.0 / 12.0);
}

// Discrete equilibrium of Eq. 7 with rho0 = 1, RT = 1/3:
//   f_eq_i = W_i [drho + 9/2 (xi.u)^2 - 3/2 |u|^2] + 3 W_i xi.u.
template <int I, typename C>
__device__ __forceinline__ C feq_i(C drho, C ux, C uy, C uz, C usq15) {
    constexpr int X = cx(I), Y = cy(I), Z = cz(I);
    C xu = C(0);
    if constexpr (X != 0) xu += C(X) * ux;
    if constexpr (Y != 0) xu += C(Y) * uy;
    if constexpr (Z != 0) xu += C(Z) * uz;
    const C w = C(w36(I)) / C(36);
    if constexpr (I == 0) return w * (drho - usq15);
    else return w * (drho + C(4.5) * xu * xu - usq15) + lin3w<C>(X * X + Y * Y + Z * Z) * xu;
}

// delta-rho = sum f, rho0 u = sum xi f (Eq. 8), rho0 = 1.
template <typename C>
__device__ __forceinline__ void moments(const C (&f)[Q], C& drho, C& jx, C& jy, C& jz) {
    C a[NPAIR], b[NPAIR];
#pragma unroll
    for (int p = 0; p < NPAIR; ++p) {
        a[p] = f[2 * p + 1] + f[2 * p + 2];
        b[p] = f[2 * p + 1] - f[2 * p + 2];
    }
    drho = f[0] + ((a[0] + a[1]) + a[2]) + (((a[3] + a[4]) + (a[5] + a[6])) + (a[7] + a[8]));
    jx = (b[0] + b[3]) + (b[4] + (b[5] + b[6]));
    jy = (b[1] + b[3]) - (b[4] - (b[7] + b[8]));
    jz = (b[2] + b[5]) - (b[6] - (b[7] - b[8]));
}

// ---------------------------------------------------------------------------
// MRT collision (Sec. II.B, RHS of Eq. 21): f <- f - M^-1 S (M f - m_eq), in place.
//
// The rows M_k are orthogonal integer polynomials of the velocity, so M^-1 =
// M^T diag(1 / |M_k|^2) and the change of f_i is sum_k M_ki g_k with
// g_k = s_k (m_k - m_eq_k) / |M_k|^2.  Rows are even or odd in xi and enter
// through the pair sums a_p and differences b_p; of these every row needs only
// the sums over the axis pairs, over the two diagonal pairs of a plane, and
// their signed counterparts.  With S_ax, S_d the sums of the axis and diagonal
// a_p and s_xy, s_xz, s_yz those of a plane:
//   k  polynomial                 m_k                           |M_k|^2   m_eq_k
//   1  19 r2 - 30                 -30 f0 - 11 S_ax + 8 S_d        2394    -11 drho + 19 j.j
//   2  (21 r4 - 53 r2 + 24) / 2    12 f0 - 4 S_ax + S_d             252    -475/63 j.j
//   4  (5 r2 - 9) x  (6 y, 8 z)   j_x - 5 b_x                       40    -2/3 j_x
//   9  3 x^2 - r2                 A + B                             36    3 j_x^2 - j.j
//  10  (3 r2 - 5)(3 x^2 - r2)     B - 2 A                           72    0
//  11  y^2 - z^2                  A' + B'                           12    j_y^2 - j_z^2
//  12  (3 r2 - 5)(y^2 - z^2)      B' - 2 A'                         24    0
//  13  x y  (14 y z, 15 x z)      a_3 - a_4                          4    j_x j_y
//  16  (y^2 - z^2) x  (17, 18)    x part of the xy pairs - xz pairs   8    0
// (A = 3 a_x - S_ax, B = S_d - 3 s_yz, A' = a_y - a_z, B' = s_xy - s_xz;
// omega_eps = omega_xx = 0, omega_epsj = -475/63, rho0 = 1; m_1 - m_eq_1 =
// 19 (S_d - f0 - j.j)).  About 165 operations a cell, against 290 with every row
// summed by itself, which bounded FP64 (64^3 135 -> 78 us) and two steps in one
// pass (lbe_pair.cuh).

// Rates of Sec. IV.A, and s_k / |M_k|^2 with the constant factors of the table.
template <typename C>
struct MrtRates {
    C s1, s2, s4, s9, s10, s13, s16;
    C c1, c2, c4, c9, c10, c11, c12, c13, c16;
};

// FIXJ: the equilibrium takes the prescribed momentum (jfx, jfy, jfz) and the
// momentum rows relax fully to it (the consistent initialisation, Sec. IV.A);
// otherwise the cell's own momentum, conserved.
template <bool FIXJ, typename C>
__device__ __forceinline__ void mrt_collide_t(C (&f)[Q], const MrtRates<C>& r, C& drho_out, C& jx_out,
                                              C& jy_out, C& jz_out, C jfx, C jfy, C jfz) {
    C a[NPAIR], b[NPAIR];
#pragma unroll
    for (int p = 0; p < NPAIR; ++p) {
        a[p] = f[2 * p + 1] + f[2 * p + 2];
        b[p] = f[2 * p + 1] - f[2 * p + 2];
    }
    const C f0 = f[0];
    const C sxy = a[3] + a[4], sxz = a[5] + a[6], syz = a[7] + a[8];
    const C sax = (a[0] + a[1]) + a[2], sd = (sxy + sxz) + syz;
    // the x, y, z parts of the diagonal pairs of a plane
    const C xxy = b[3] + b[4], xxz = b[5] + b[6];
    const C yxy = b[3] - b[4], yyz = b[7] + b[8];
    const C zxz = b[5] - b[6], zyz = b[7] - b[8];
    const C drho = f0 + (sax + sd);
    const C jx = b[0] + (xxy + xxz), jy = b[1] + (yxy + yyz), jz = b[2] + (zxz + zyz);
    drho_out = drho;
    jx_out = jx;
    jy_out = jy;
    jz_out = jz;
    const C ex = FIXJ ? jfx : jx, ey = FIXJ ? jfy : jy, ez = FIXJ ? jfz : jz;  // momentum of m_eq
    // (products that meet a plain addition go through mul_rn, so that every
    // kernel this is inlined in rounds alike)
    const C xx = mul_rn(ex, ex), yy = mul_rn(ey, ey);
    const C jj = fma(ez, ez, xx + yy);

    const C g1 = mul_rn(r.c1, ((sd - f0) - jj));
    const C g2 = mul_rn(r.c2, fma(C(475.0 / 63.0), jj, fma(C(12), f0, fma(C(-4), sax, sd))));
    const C A9 = fma(C(3), a[0], -sax), B9 = fma(C(-3), syz, sd);
    const C g9 = mul_rn(r.c9, fma(C(-3), xx, (A9 + B9) + jj));
    const C g10 = mul_rn(r.c10, fma(C(-2), A9, B9));
    const C A11 = a[1] - a[2], B11 = sxy - sxz;
    const C g11 = mul_rn(r.c11, fma(ez, ez, (A11 + B11) - yy));
    const C g12 = mul_rn(r.c12, fma(C(-2), A11, B11));
    const C g13 = mul_rn(r.c13, fma(-ex, ey, a[3] - a[4]));
    const C g14 = mul_rn(r.c13, fma(-ey, ez, a[7] - a[8]));
    const C g15 = mul_rn(r.c13, fma(-ex, ez, a[5] - a[6]));
    // c4 carries the factor 5 of j - 5 b
    C g4, g6, g8;
    if constexpr (FIXJ) {
        g4 = mul_rn(r.c4, fma(C(0.2), fma(C(2.0 / 3.0), ex, jx), -b[0]));
        g6 = mul_rn(r.c4, fma(C(0.2), fma(C(2.0 / 3.0), ey, jy), -b[1]));
        g8 = mul_rn(r.c4, fma(C(0.2), fma(C(2.0 / 3.0), ez, jz), -b[2]));
    } else {
        g4 = mul_rn(r.c4, fma(C(1.0 / 3.0), jx, -b[0]));
        g6 = mul_rn(r.c4, fma(C(1.0 / 3.0), jy, -b[1]));
        g8 = mul_rn(r.c4, fma(C(1.0 / 3.0), jz, -b[2]));
    }
    const C g16 = mul_rn(r.c16, xxy - xxz), g17 = mul_rn(r.c16, yyz - yxy), g18 = mul_rn(r.c16, zxz - zyz);

    // back transform: df_i = sum_k M_ki g_k, even part e and odd part o of a pair
    f[0] = f0 - fma(C(-30), g1, C(12) * g2);
    C e[NPAIR], o[NPAIR];
    const C eax = fma(C(-11), g1, C(-4) * g2);
    const C h9 = fma(C(-2), g10, g9), h11 = fma(C(-2), g12, g11);
    e[0] = fma(C(2), h9, eax);
    e[1] = (eax - h9) + h11;
    e[2] = (eax - h9) - h11;
    const C ed = fma(C(8), g1, g2);
    const C k9 = g9 + g10, k11 = g11 + g12;
    const C exy = (ed + k9) + k11, exz = (ed + k9) - k11, eyz = fma(C(-2), k9, ed);
    e[3] = exy + g13;
    e[4] = exy - g13;
    e[5] = exz + g15;
    e[6] = exz - g15;
    e[7] = eyz + g14;
    e[8] = eyz - g14;
    o[0] = mul_rn(C(-4), g4);
    o[1] = mul_rn(C(-4), g6);
    o[2] = mul_rn(C(-4), g8);
    C x1 = g4 + g16, x2 = g4 - g16, y1 = g6 - g17, y2 = g6 + g17, z1 = g8 + g18, z2 = g8 - g18;
    if constexpr (FIXJ) {
        // the momentum rows (M_3,5,7 = xi_x, xi_y, xi_z) relaxed with rate 1, |M_3|^2 = 10
        const C gx = mul_rn(jx - jfx, C(0.1)), gy = mul_rn(jy - jfy, C(0.1)), gz = mul_rn(jz - jfz, C(0.1));
        o[0] += gx;
        o[1] += gy;
        o[2] += gz;
        x1 += gx;
        x2 += gx;
        y1 += gy;
        y2 += gy;
        z1 += gz;
        z2 += gz;
    }
    o[3] = x1 + y1;
    o[4] = x1 - y1;
    o[5] = x2 + z1;
    o[6] = x2 - z1;
    o[7] = y2 + z2;
    o[8] = y2 - z2;
#pragma unroll
    for (int p = 0; p < NPAIR; ++p) {
        f[2 * p + 1] -= e[p] + o[p];
        f[2 * p + 2] -= e[p] - o[p];
    }
}

// ---------------------------------------------------------------------------
// MRT collision of 2-byte storage, every row of M summed by itself.  The state of
// such a run is its storage rounding noise: any other order of the FP32
// operations reshuffles it, and E of a 32^3 BF16 run moves by 5e-3.  So these
// runs keep this order, and with it their results bit for bit, at 214 us a
// 256^3 FP16 step where the order of mrt_collide_t takes 184.
//
// Moment rows of Sec. II.B as integer polynomials of the velocity.
__host__ __device__ constexpr int mrow(int k, int x, int y, int z) {
    const int r2 = x * x + y * y + z * z;
    switch (k) {
        case 0: return 1;
        case 1: return 19 * r2 - 30;
        case 2: return (21 * r2 * r2 - 53 * r2 + 24) / 2;
        case 3: return x;
        case 4: return (5 * r2 - 9) * x;
        case 5: return y;
        case 6: return (5 * r2 - 9) * y;
        case 7: return z;
        case 8: return (5 * r2 - 9) * z;
        case 9: return 3 * x * x - r2;
        case 10: return (3 * r2 - 5) * (3 * x * x - r2);
        case 11: return y * y - z * z;
        case 12: return (3 * r2 - 5) * (y * y - z * z);
        case 13: return x * y;
        case 14: return y * z;
        case 15: return x * z;
        case 16: return (y * y - z * z) * x;
        case 17: return (z * z - x * x) * y;
        default: return (x * x - y * y) * z;
    }
}
// Squared norm of row k over the 19 velocities.
__host__ __device__ constexpr int mnorm(int k) {
    int s = 0;
    for (int i = 0; i < Q; ++i) {
        int v = mrow(k, cx(i), cy(i), cz(i));
        s += v * v;
    }
    return s;
}
// Non-conserved rows whose polynomial is even / odd in xi.
__host__ __device__ constexpr int even_row(int j) {
    return j == 0 ? 1 : j == 1 ? 2 : j == 2 ? 9 : j == 3 ? 10 : j == 4 ? 11 : j == 5 ? 12 : j == 6 ? 13
         : j == 7 ? 14 : 15;
}
__host__ __device__ constexpr int odd_row(int j) {
    return j == 0 ? 4 : j == 1 ? 6 : j == 2 ? 8 : j == 3 ? 16 : j == 4 ? 17 : 18;
}
constexpr int NEVEN = 9;
constexpr int NODD = 6;

template <int K, typename C>
__device__ __forceinline__ C rate(const MrtRates<C>& r) {
    if constexpr (K == 1) return r.s1;
    else if constexpr (K == 2) return r.s2;
    else if constexpr (K == 4 || K == 6 || K == 8) return r.s4;
    else if constexpr (K == 9 || K == 11) return r.s9;
    else if constexpr (K == 10 || K == 12) return r.s10;
    else if constexpr (K == 13 || K == 14 || K == 15) return r.s13;
    else return r.s16;
}

// Equilibrium moments (Sec. II.B with omega_eps = omega_xx = 0,
// omega_epsj = -475/63, rho0 = 1).  Slot 9 holds 3 p_xx.
template <int K, typename C>
__device__ __forceinline__ C meq(C drho, C jx, C jy, C jz, C jj) {
    if constexpr (K == 1) return C(-11) * drho + C(19) * jj;
    else if constexpr (K == 2) return C(-475.0 / 63.0) * jj;
    else if constexpr (K == 4) return C(-2.0 / 3.0) * jx;
    else if constexpr (K == 6) return C(-2.0 / 3.0) * jy;
    else if constexpr (K == 8) return C(-2.0 / 3.0) * jz;
    else if constexpr (K == 9) return C(2) * jx * jx - (jy * jy + jz * jz);
    else if constexpr (K == 11) return jy * jy - jz * jz;
    else if constexpr (K == 13) return jx * jy;
    else if constexpr (K == 14) return jy * jz;
    else if constexpr (K == 15) return jx * jz;
    else return C(0);  // rows 10, 12 (omega_xx = 0) and 16-18
}

// One MRT collision in place (RHS of Eq. 21): f <- f - M^-1 S (M f - m_eq).
// M is orthogonal, so M^-1 = M^T diag(1/|M_k|^2); rows are even or odd in xi,
// so the work splits into the pair sums a_p = f_{2p+1} + f_{2p+2} (even rows)
// and differences b_p = f_{2p+1} - f_{2p+2} (odd rows).
// FIXJ: the equilibrium takes the prescribed momentum (jfx, jfy, jfz) and the
// momentum rows relax fully to it (the consistent initialisation, Sec. IV.A);
// otherwise the cell's own momentum, conserved.
template <bool FIXJ, typename C>
__device__ __forceinline__ void mrt_collide_rows(C (&f)[Q], const MrtRates<C>& r, C& drho_out, C& jx_out,
                                              C& jy_out, C& jz_out, C jfx, C jfy, C jfz) {
    C a[NPAIR], b[NPAIR];
#pragma unroll
    for (int p = 0; p < NPAIR; ++p) {
        a[p] = f[2 * p + 1] + f[2 * p + 2];
        b[p] = f[2 * p + 1] - f[2 * p + 2];
    }
    const C f0 = f[0];
    const C drho = f0 + ((a[0] + a[1]) + a[2]) + (((a[3] + a[4]) + (a[5] + a[6])) + (a[7] + a[8]));
    const C jx = (b[0] + b[3]) + (b[4] + (b[5] + b[6]));
    const C jy = (b[1] + b[3]) - (b[4] - (b[7] + b[8]));
    const C jz = (b[2] + b[5]) - (b[6] - (b[7] - b[8]));
    drho_out = drho;
    jx_out = jx;
    jy_out = jy;
    jz_out = jz;
    const C jxe = FIXJ ? jfx : jx, jye = FIXJ ? jfy : jy, jze = FIXJ ? jfz : jz;
    const C jj = jxe * jxe + jye * jye + jze * jze;
    // FIXJ: (m - m_eq) / |M_k|^2 of the momentum rows at rate 1 (|M_3|^2 = 10)
    [[maybe_unused]] const C gjx = (jx - jfx) * C(0.1), gjy = (jy - jfy) * C(0.1), gjz = (jz - jfz) * C(0.1);

    C ge[NEVEN], go[NODD];
    static_for<0, NEVEN>([&](auto jc) {
        constexpr int J = decltype(jc)::value;
        constexpr int K = even_row(J);
        C m = C(mrow(K, 0, 0, 0)) * f0;
        static_for<0, NPAIR>([&](auto pc) {
            constexpr int P = decltype(pc)::value;
            constexpr int c = mrow(K, pair_x(P), pair_y(P), pair_z(P));
            if constexpr (c == 1) m += a[P];
            else if constexpr (c == -1) m -= a[P];
            else if constexpr (c != 0) m += C(c) * a[P];
        });
        ge[J] = rate<K>(r) * (m - meq<K>(drho, jxe, jye, jze, jj)) * (C(1) / C(mnorm(K)));
    });
    static_for<0, NODD>([&](auto jc) {
        constexpr int J = decltype(jc)::value;
        constexpr int K = odd_row(J);
        C m = C(0);
        static_for<0, NPAIR>([&](auto pc) {
            constexpr int P = decltype(pc)::value;
            constexpr int c = mrow(K, pair_x(P), pair_y(P), pair_z(P));
            if constexpr (c == 1) m += b[P];
            else if constexpr (c == -1) m -= b[P];
            else if constexpr (c != 0) m += C(c) * b[P];
        });
        go[J] = rate<K>(r) * (m - meq<K>(drho, jxe, jye, jze, jj)) * (C(1) / C(mnorm(K)));
    });
    // back transform: df_i = sum_k M_k,i g_k
    {
        C d0 = C(0);
        static_for<0, NEVEN>([&](auto jc) {
            constexpr int J = decltype(jc)::value;
            constexpr int c = mrow(even_row(J), 0, 0, 0);
            if constexpr (c != 0) d0 += C(c) * ge[J];
        });
        f[0] = f0 - d0;
    }
    static_for<0, NPAIR>([&](auto pc) {
        constexpr int P = decltype(pc)::value;
        C e = C(0), o = C(0);
        static_for<0, NEVEN>([&](auto jc) {
            constexpr int J = decltype(jc)::value;
            constexpr int c = mrow(even_row(J), pair_x(P), pair_y(P), pair_z(P));
            if constexpr (c == 1) e += ge[J];
            else if constexpr (c == -1) e -= ge[J];
            else if constexpr (c != 0) e += C(c) * ge[J];
        });
        static_for<0, NODD>([&](auto jc) {
            constexpr int J = decltype(jc)::value;
            constexpr int c = mrow(odd_row(J), pair_x(P), pair_y(P), pair_z(P));
            if constexpr (c == 1) o += go[J];
            else if constexpr (c == -1) o -= go[J];
            else if constexpr (c != 0) o += C(c) * go[J];
        });
        if constexpr (FIXJ) {
            // the momentum rows (M_3,5,7 = xi_x, xi_y, xi_z) relaxed with rate 1
            if constexpr (pair_x(P) != 0) o += C(pair_x(P)) * gjx;
            if constexpr (pair_y(P) != 0) o += C(pair_y(P)) * gjy;
            if constexpr (pair_z(P) != 0) o += C(pair_z(P)) * gjz;
        }
        f[2 * P + 1] -= e + o;
        f[2 * P + 2] -= e - o;
    });
}

// The collision of storage type S.
template <typename S, bool FIXJ, typename C>
__device__ __forceinline__ void mrt_collide_as(C (&f)[Q], const MrtRates<C>& r, C jfx = C(0), C jfy = C(0), C jfz = C(0)) {
    C drho, jx, jy, jz;
    if constexpr (sizeof(S) == 2) mrt_collide_rows<FIXJ>(f, r, drho, jx, jy, jz, jfx, jfy, jfz);
    else mrt_collide_t<FIXJ>(f, r, drho, jx, jy, jz, jfx, jfy, jfz);
}

// Periodic neighbour of coordinate v in [0, n).
__device__ __forceinline__ int wrap_inc(int v, int n) { return v + 1 == n ? 0 : v + 1; }
__device__ __forceinline__ int wrap_dec(int v, int n) { return v == 0 ? n - 1 : v - 1; }

}  // namespace kin
