// lbm_fx.cuh -- the BGK relaxation of the FP64 form (Eqs. LBM_Equation, LBM_EQ,
// Forcing) in 64-bit fixed point.
//
// The populations of a fluid near rest are below 1/2 and their rounding errors
// absolute (2^-58 for the diagonals), so units of 2^-62 ... 2^-64 hold every
// quantity of the update more precisely than FP64 does: sums are exact, and a
// product (the high half of a 64 x 64-bit multiplication) costs a third of an
// FP64 multiply on GB300, a sum a tenth.  With A = omega rho u / 12, G = kf F /
// 12, H = A + G and V = u / eps the update of Sec. 3.2.2, divided by 36, is
//   E' = omega rho / 36 - (Dx + Dy + Dz)/3,  D_a = 3/2 (H_a + G_a) V_a,
//   X_ab = 3 (H_a V_b + G_b V_a),
//   f0  <- f0 - omega f0 + 12 E',
//   f+-a <- f - omega f + 2 (E' + D_a) +- 2 H_a,
//   f+-a+-b <- f - omega f + E' + D_a + D_b +- X_ab +- H_a +- H_b,
// which needs no multiplication per direction beyond omega f.  Cells
// outside the ranges below (populations about twice those at rest, or below
// 2^-10) take the FP64 path, as do non-finite ones.
//
// A rounding of one sign would add up over cells and steps, so the sums that the
// update conserves are kept: f_0 is what the other 18 leave of rho, exactly, and
// f_ext and the odd part H, which carry the momentum, are rounded to nearest (zero
// stays zero), and the halves of the final rounding cancel over the populations.
// Mean error of a cell's mass and momentum per step against exact arithmetic, with
// and without f_ext, tau 0.5045 to 3, 200,000 cells: below 8e-20 and 3e-20, the
// noise of that mean (FP64: 7.5e-17 and 7e-20).  The even products round down.
#pragma once
#include "dps_internal.cuh"

namespace dps {

// v in [2^-10, 1) in units of 2^-62, exactly: its 53 bits moved up by 0 to 9
__host__ __device__ __forceinline__ i64 fx_q62(u64 b) {
    return (i64)(((b & 0x000fffffffffffffull) | 0x0010000000000000ull) << (((u32)(b >> 52) + 11) & 31));
}
__host__ __device__ __forceinline__ double fx_signed_to_double(i64 v, int frac) {
    return fx_with_sign(fx_to_double((u64)(v < 0 ? -v : v), frac), v);
}
// v >= 2^32, units of 2^-frac, rounded to double (halves up; EVEN: halves to even)
template <bool EVEN = false>
__host__ __device__ __forceinline__ double fx_positive_to_double(u64 v, int frac) {
#ifdef __CUDA_ARCH__
    const u32 hi = (u32)(v >> 32), lo = (u32)v;
    const int lz = __clz((int)hi);
    const u32 h = __funnelshift_l(lo, hi, lz), l = lo << lz;
#else
    const int lz = fx_clz(v);
    const u32 h = (u32)(v << lz >> 32), l = (u32)(v << lz);
#endif
    const u32 up = EVEN ? (l & 0x7ffu) + ((l >> 11) & 1) > 0x400u : (l >> 10) & 1;
    return fx_double((((u64)h << 32 | l) >> 11) + up + ((u64)((u32)(1022 + 63 - frac - lz) << 20) << 32));
}
// a b 2^-64 for a, b >= 0, rounded down, the product of the low halves left
// out: at most 3 units low, 1.25 in the mean
__host__ __device__ __forceinline__ u64 fx_mulhi_short(u64 a, u64 b) {
    const u32 ah = (u32)(a >> 32), al = (u32)a, bh = (u32)(b >> 32), bl = (u32)b;
    return (u64)ah * bh + (((u64)ah * bl) >> 32) + (((u64)al * bh) >> 32);
}
// a b 2^-63 (below 2^63) rounded to nearest
__host__ __device__ __forceinline__ i64 fx_mul_near63(i64 a, i64 b) {
    const u64 lo = (u64)a * (u64)b;
    return fx_mulhi_s(a, b) * 2 + (i64)(lo >> 63) + (i64)((lo >> 62) & 1);
}
__host__ __device__ __forceinline__ u32 fx_abs_hi(u64 b) { return (u32)(b >> 32) & 0x7fffffffu; }

// populations in units of 2^-62 and their exact moments; false when one is
// below 2^-10, or not below 1/2 (f_0), 1/8 (along an axis), 1/16 (along a
// diagonal: their sum stays below 2), or not finite
__host__ __device__ __forceinline__ bool fx_populations(const u64 b[Q], i64 f[Q], i64 &rho, i64 j[3]) {
    int axis = 0, diag = 0, low = (int)(b[0] >> 32);  // high words: ordered like the values
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int q = 1; q < Q; ++q) {
        const int h = (int)(b[q] >> 32);
        if (CX(q) * CX(q) + CY(q) * CY(q) + CZ(q) * CZ(q) == 1) axis = axis > h ? axis : h;
        else diag = diag > h ? diag : h;
        low = low < h ? low : h;
    }
    if (!(low >= 0x3f500000 && (int)(b[0] >> 32) < 0x3fe00000 && axis < 0x3fc00000 && diag < 0x3fb00000)) return false;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int q = 0; q < Q; ++q) f[q] = fx_q62(b[q]);
    rho = f[0];
    j[0] = j[1] = j[2] = 0;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int k = 1; k <= 9; ++k) {
        rho += f[k] + f[k + 9];
        const i64 d = f[k] - f[k + 9];
        if (CX(k) != 0) j[0] += CX(k) > 0 ? d : -d;
        if (CY(k) != 0) j[1] += CY(k) > 0 ? d : -d;
        if (CZ(k) != 0) j[2] += CZ(k) > 0 ? d : -d;
    }
    return true;
}

// box constants of the relaxation
__host__ __device__ inline FxFluid fx_fluid(double omega, double kf, const double fb[3]) {
    FxFluid x;
    std::memset(&x, 0, sizeof x);
    x.ok = omega > 0.0 && omega < 2.0 && kf > 0.0 && kf < 1.0 && fabs(fb[0]) < 0.125 && fabs(fb[1]) < 0.125 &&
           fabs(fb[2]) < 0.125;
    if (!x.ok) return x;
    x.om = (u64)fx_from_pos(omega, 60) * 8;
    const u64 o = (u64)fx_from_pos(omega, 60), k = (u64)fx_from_pos(kf, 60);
    // omega/12, omega/36, kf/12 in units of 2^-64 to nearest: 16/12 = 4/3 and 16/36 = 4/9 of the 2^-60 value
    x.om12 = o / 3 * 4 + ((o % 3) * 4 + 1) / 3;
    x.om36 = o / 9 * 4 + ((o % 9) * 4 + 4) / 9;
    x.kf12 = k / 3 * 4 + ((k % 3) * 4 + 1) / 3;
    for (int a = 0; a < 3; ++a) x.fb[a] = (i64)llrint(fb[a] * 0x1p66);
    return x;
}

// 1/(rho eps) = R 2^(lz-64), R in (2^62, 2^63] (Newton from a single-precision
// seed); rho eps in (1/16, 2), both in units of 2^-62
__host__ __device__ __forceinline__ u64 fx_recip(i64 rho, i64 e62, int &lz) {
    u64 P = fx_mulhi((u64)rho << 1, (u64)e62 << 1);  // 2^-62
    lz = fx_clz(P);
    P <<= lz;
    u32 Y = (u32)(fx_rcp_seed((float)(u32)(P >> 32) * 0x1p-32f) * 0x1p30f);
    Y = Y > 0x7fffffffu ? 0x7fffffffu : Y;
    const i64 e1 = (i64)((1ull << 63) - fx_mulhi(P, (u64)Y << 33));  // y (1 + e1 + e1^2)
    const i64 f1 = (i64)(int)(e1 >> 12);
    const i64 c1 = e1 + ((f1 * f1) >> 39);
    return ((u64)Y << 32) + (u64)(((c1 >> 32) * (i64)Y) * 2) + (((u64)(u32)c1 * Y) >> 31);
}

// omega = 1/tau_e of a cell (Eq. tau_e) from its populations f and rho (2^-62),
// J = rho u (2^-66) and V = u/eps (2^-60).  The non-equilibrium flux Q_ab is
// exact integer sums and three-half products; square roots and divisions are
// FP64 (tau_* of the Eilers viscosity, tau_t of Smagorinsky, in the
// cancellation-free form).
__host__ __device__ __forceinline__ double fx_omega_cell(const i64 f[Q], i64 rho, const i64 J[3], const i64 V[3],
                                                         i64 ir, double e, double tau, int eilers, int smag) {
    double ts = tau;
    if (eilers) {
        double r = (1.0 - e) * (1.0 / 0.64);
        r = r < 0.0 ? 0.0 : (r > 0.9 ? 0.9 : r);
        const double a = 1.0 + (1.25 * 0.64) * r / (1.0 - r);
        ts = 0.5 + (tau - 0.5) * (a * a);
    }
    if (!smag) return 1.0 / ts;
    const i64 iso = fx_mulhi_s(rho, 6148914691236517205ll);  // rho/3
    i64 P[6] = {-iso, -iso, -iso, 0, 0, 0};                  // xx yy zz xy xz yz
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int k = 1; k <= 9; ++k) {
        const i64 p = f[k] + f[k + 9];
        if (CX(k) != 0) P[0] += p;
        if (CY(k) != 0) P[1] += p;
        if (CZ(k) != 0) P[2] += p;
        if (CX(k) * CY(k) != 0) P[3] += CX(k) * CY(k) > 0 ? p : -p;
        if (CX(k) * CZ(k) != 0) P[4] += CX(k) * CZ(k) > 0 ? p : -p;
        if (CY(k) * CZ(k) != 0) P[5] += CY(k) * CZ(k) > 0 ? p : -p;
    }
    double q[6];
    q[0] = fx_signed_to_double(P[0] - fx_mulhi_s(J[0], V[0]), 62);
    q[1] = fx_signed_to_double(P[1] - fx_mulhi_s(J[1], V[1]), 62);
    q[2] = fx_signed_to_double(P[2] - fx_mulhi_s(J[2], V[2]), 62);
    q[3] = fx_signed_to_double(P[3] - fx_mulhi_s(J[0], V[1]), 62);
    q[4] = fx_signed_to_double(P[4] - fx_mulhi_s(J[0], V[2]), 62);
    q[5] = fx_signed_to_double(P[5] - fx_mulhi_s(J[1], V[2]), 62);
    const double q2 = q[0] * q[0] + q[1] * q[1] + q[2] * q[2] + 2.0 * (q[3] * q[3] + q[4] * q[4] + q[5] * q[5]);
    // 2 C_S^2 Qbar / (rho c_s^4)
    const double x = (2 * 0.01 * 9) * sqrt(2.0 * q2) * fx_positive_to_double((u64)ir, 62);
    const double y = 2.0 * (sqrt(ts * ts + x) + ts);
    return y / (ts * y + x);  // 1/(tau_* + x/y)
}

// One cell: b the bits of the populations, e = eps_f, fp = f_pf; f receives the
// post-collision populations.  VISC: omega from the cell's own tau_e (vmode bit
// 0 Eilers, bit 1 Smagorinsky), else the box's.  False: outside the range,
// nothing is written.
template <bool VISC>
__host__ __device__ __forceinline__ bool fx_relax(const u64 b[Q], double e, double fp0, double fp1, double fp2,
                                                  const FxFluid &xb, double tau, int vmode, double out[Q]) {
    FxFluid x = xb;
    i64 f[Q], rho, j[3];
    const u64 eb = fx_bits(e), p0 = fx_bits(fp0), p1 = fx_bits(fp1), p2 = fx_bits(fp2);
    // 1/8 < eps <= 1, |f_pf| < 1/8
    if (!(eb > 0x3fc0000000000000ull && eb <= 0x3ff0000000000000ull && fx_abs_hi(p0) < 0x3fc00000u &&
          fx_abs_hi(p1) < 0x3fc00000u && fx_abs_hi(p2) < 0x3fc00000u && x.ok))
        return false;
    if (!fx_populations(b, f, rho, j)) return false;
    const i64 e62 = fx_from_pos(e, 62);
    i64 F[3] = {fx_from(fp0, 65), fx_from(fp1, 65), fx_from(fp2, 65)}, J[3];
    // f_ext = f_pf + eps_f f_b (|.| < 1/4), 2^-65; 1/2 < rho < 2, |j + F/2| < 1/8 per component
    const i64 lim = 1ll << 59;
    bool in = rho > (1ll << 61);
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int a = 0; a < 3; ++a) {
        F[a] += fx_mul_near63(e62, x.fb[a]);
        const i64 t = j[a] + (F[a] >> 4);
        in = in && t < lim && t > -lim;
        J[a] = (i64)((u64)j[a] * 16 + (u64)F[a]);  // rho u = j + F/2, 2^-66
    }
    if (!in) return false;
    int lz;
    const u64 R = fx_recip(rho, e62, lz);
    i64 V[3];  // u/eps = (j + F/2)/(rho eps), 2^-60, |.| < 2
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int a = 0; a < 3; ++a) V[a] = fx_mulhi_s(J[a], (i64)(R >> 1)) >> (5 - lz);
    if (VISC && vmode) {
        const i64 ir = (i64)(fx_mulhi((u64)e62, R) << lz);  // 1/rho, 2^-62, < 2
        const double om = fx_omega_cell(f, rho, J, V, ir, e, tau, vmode & 1, vmode & 2);
        if (!(om > 0.0 && om < 2.0)) return false;
        const u64 o = (u64)fx_from_pos(om, 60), k = (1ull << 60) - (o >> 1);  // omega, 1 - omega/2
        x.om = o * 8;
        x.om12 = o + fx_mulhi(o, 0x5555555555555555ull);
        x.om36 = fx_mulhi(o, 0x71c71c71c71c71c7ull);
        x.kf12 = k + fx_mulhi(k, 0x5555555555555555ull);
    }
    i64 H[3], O[3], G[3];
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int a = 0; a < 3; ++a) {
        // omega rho u/12 + kf F/12 = h 2^-66, rounded once to 2^-63
        const u64 jl = (u64)J[a] * x.om12, fl = (u64)F[a] * x.kf12;
        const i64 g = fx_mulhi_s(F[a], (i64)x.kf12);  // 2^-65
        const i64 h = fx_mulhi_s(J[a], (i64)x.om12) + 2 * g + (i64)(fl >> 63) + (i64)(jl + 2 * fl < jl);
        O[a] = (h + 4) >> 3;
        H[a] = h * 2;  // 2^-67
        G[a] = g * 4;
    }
    // the even parts in units of 2^-63
    i64 D[3], S = 0;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int a = 0; a < 3; ++a) {
        const i64 p = fx_mulhi_s(H[a] + G[a], V[a]);
        D[a] = p + (p >> 1);
        S += D[a];
    }
    const i64 E = (i64)fx_mulhi(x.om36, (u64)rho << 1) - fx_mulhi_s(S, 6148914691236517205ll);
    const i64 Xxy = 3 * (fx_mulhi_s(H[0], V[1]) + fx_mulhi_s(G[1], V[0]));
    const i64 Xxz = 3 * (fx_mulhi_s(H[0], V[2]) + fx_mulhi_s(G[2], V[0]));
    const i64 Xyz = 3 * (fx_mulhi_s(H[1], V[2]) + fx_mulhi_s(G[2], V[1]));
    // f - omega f + ...; f_0 takes what the others leave of rho (the even parts
    // of the nine pairs add to 12 E + 6 S a side)
    i64 v[Q];
    u64 rest = (u64)f[0] * 2 - (u64)E * 24 - (u64)S * 12 - 1;
    int low = 0x7fffffff;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int k = 1; k <= 9; ++k) {
        i64 ev = E, od = 0;
        if (CX(k) != 0) { ev += D[0]; od += CX(k) > 0 ? O[0] : -O[0]; }
        if (CY(k) != 0) { ev += D[1]; od += CY(k) > 0 ? O[1] : -O[1]; }
        if (CZ(k) != 0) { ev += D[2]; od += CZ(k) > 0 ? O[2] : -O[2]; }
        if (CX(k) * CY(k) != 0) ev += CX(k) * CY(k) > 0 ? Xxy : -Xxy;
        if (CX(k) * CZ(k) != 0) ev += CX(k) * CZ(k) > 0 ? Xxz : -Xxz;
        if (CY(k) * CZ(k) != 0) ev += CY(k) * CZ(k) > 0 ? Xyz : -Xyz;
        if (CX(k) * CX(k) + CY(k) * CY(k) + CZ(k) * CZ(k) == 1) {
            ev *= 2;
            od *= 2;
        }
        const i64 p = (i64)fx_mulhi_short(x.om, (u64)f[k] << 2), r = (i64)fx_mulhi_short(x.om, (u64)f[k + 9] << 2);
        rest += (u64)(p + r);
        // the halves of a pair round up below, or down with one unit less: five
        // pairs up and four down, and f_0 with its halves to even one unit less
        if (!(k & 1)) ev -= 1;
        v[k] = f[k] * 2 - p + ev + od;
        v[k + 9] = f[k + 9] * 2 - r + ev - od;
        const int a = (int)(v[k] >> 32), c = (int)(v[k + 9] >> 32);
        low = low < a ? low : a;
        low = low < c ? low : c;
    }
    v[0] = (i64)rest;
    low = low < (int)(v[0] >> 32) ? low : (int)(v[0] >> 32);
    if (low > 0) {
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
        for (int q = 1; q < Q; ++q) out[q] = fx_positive_to_double((u64)v[q], 63);
        out[0] = fx_positive_to_double<true>((u64)v[0], 63);
    } else {  // a population at or below zero
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
        for (int q = 0; q < Q; ++q) out[q] = fx_signed_to_double(v[q], 63);
    }
    return true;
}

}  // namespace dps
