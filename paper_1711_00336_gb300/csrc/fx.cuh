// fx.cuh -- the sphere-pair geometry and the lubrication coefficients of the
// FP64 form in 64-bit integer arithmetic.
//
// An SM of GB300 retires an FP64 warp instruction every ~19 cycles and two to
// four 32-bit integer ones per cycle, so a 64-bit fixed-point product (four
// 32-bit multiply-adds and their carries) costs a third of one FP64 multiply
// and an addition a tenth.  The separation, the unit normal, the gap, the
// logarithm and the reciprocal of a lubrication pair therefore run on 64-bit
// integers with 58 to 63 fraction bits, each value scaled so that its leading
// bits are used.  Against exact arithmetic the coefficients of a pair of spheres
// are 2 to 40 times as close as FP64's (as close next to the origin of a box of
// 512 cells or more); those of a wall, whose gap is taken in FP64, 2 to 3 times
// (largest error of 20,000: 2.0e-16 and 5.8e-16).  The reciprocal and the
// reciprocal square root are Newton's iteration from a single-precision seed, the
// logarithm a table of 128 reciprocals and the Taylor series of ln(1 + u).
//
// Every function is host and device code with the same results up to the
// single-precision seeds, whose last bits do not survive the iterations'
// rounding above 2^-57.
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>

#include "log_table.cuh"

namespace dps {

typedef unsigned long long u64;
typedef long long i64;
typedef unsigned int u32;

struct FxLogRow {
    i64 C, T;
};
static __device__ const FxLogRow fx_log_dev[128] = {DPS_FX_LOG_ROWS};
static const FxLogRow fx_log_host[128] = {DPS_FX_LOG_ROWS};

__host__ __device__ __forceinline__ u64 fx_mulhi(u64 a, u64 b) {
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (u64)(((unsigned __int128)a * b) >> 64);
#endif
}
__host__ __device__ __forceinline__ i64 fx_mulhi_s(i64 a, i64 b) {
#ifdef __CUDA_ARCH__
    return __mul64hi(a, b);
#else
    return (i64)(((__int128)a * b) >> 64);
#endif
}
__host__ __device__ __forceinline__ int fx_mulhi32(int a, int b) { return (int)(((i64)a * b) >> 32); }
__host__ __device__ __forceinline__ int fx_clz(u64 v) {  // 64 for 0
#ifdef __CUDA_ARCH__
    return __clzll((i64)v);
#else
    return v ? __builtin_clzll(v) : 64;
#endif
}
__host__ __device__ __forceinline__ u64 fx_bits(double v) {
#ifdef __CUDA_ARCH__
    return (u64)__double_as_longlong(v);
#else
    u64 b;
    std::memcpy(&b, &v, 8);
    return b;
#endif
}
__host__ __device__ __forceinline__ double fx_double(u64 b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((i64)b);
#else
    double v;
    std::memcpy(&v, &b, 8);
    return v;
#endif
}
// seeds: single precision, relative error below 2^-21
__host__ __device__ __forceinline__ float fx_rsqrt_seed(float x) {
#ifdef __CUDA_ARCH__
    return rsqrtf(x);
#else
    return 1.0f / std::sqrt(x);
#endif
}
__host__ __device__ __forceinline__ float fx_rcp_seed(float x) {
#ifdef __CUDA_ARCH__
    return __fdividef(1.0f, x);
#else
    return 1.0f / x;
#endif
}

// v >= 0 in units of 2^-frac, bits below dropped; |v| < 2^(62 - frac)
__host__ __device__ __forceinline__ i64 fx_from_pos(double v, int frac) {
    const u64 b = fx_bits(v);
    const int e = (int)(b >> 52) - 1023;
    const u64 m = ((b & 0x000fffffffffffffull) | 0x0010000000000000ull) << 10;  // v = m 2^(e-62)
    int sh = 62 - frac - e;
    sh = sh > 63 ? 63 : (sh < 0 ? 0 : sh);
    return (i64)(m >> sh);
}
__host__ __device__ __forceinline__ i64 fx_from(double v, int frac) {
    const i64 m = fx_from_pos(fx_double(fx_bits(v) & 0x7fffffffffffffffull), frac);
    return (i64)fx_bits(v) < 0 ? -m : m;
}
// a 64-bit magnitude v (units of 2^-frac) rounded to double
__host__ __device__ __forceinline__ double fx_to_double(u64 v, int frac) {
    const int lz = fx_clz(v);
    const u64 m = v << (lz & 63);
    const u64 r = (m >> 11) + ((m >> 10) & 1);  // 53 bits, the hidden one carries into the exponent
    const u64 b = ((u64)(u32)(1022 + 63 - lz - frac) << 52) + r;
    return v ? fx_double(b) : 0.0;
}

// the sign of s on v >= 0, as bits (a negation would be an FP64 instruction)
__host__ __device__ __forceinline__ double fx_with_sign(double v, i64 s) {
    return fx_double(fx_bits(v) | ((u64)s & 0x8000000000000000ull));
}
// the particle constants of the pair path: the radius in units of 2^-56 and
// 1/d in units of 2^-58 (1/4 <= d < 8: both exact to below an FP64 rounding)
__host__ __device__ __forceinline__ i64 fx_radius(double d) { return fx_from_pos(0.5 * d, 56); }
__host__ __device__ __forceinline__ i64 fx_inv_d(double d) {
    // 2^58/d from the FP64 quotient and its remainder
    const double q = 1.0 / d;
    return (i64)fx_from_pos(q, 58) + (i64)(fma(-q, d, 1.0) * q * 0x1p58);
}

// box constants of the pair path
struct FxBox {
    i64 hc, hmin; // h_c, h_min in units of 2^-56
    int frac;     // positions in units of 2^-frac
    u64 hmin_m;   // h_min = hmin_m 2^hmin_e, leading bit set
    int hmin_e;
    u64 c_m;      // (pi/2) mu = c_m 2^c_e, leading bit set
    int c_e;
    int ok;       // the box's sizes lie in the range of the integer path
};
__host__ __device__ inline void fx_split(double v, u64 &m, int &e) {  // v > 0, normal
    const u64 b = fx_bits(v);
    m = ((b & 0x000fffffffffffffull) | 0x0010000000000000ull) << 11;
    e = (int)(b >> 52) - 1023 - 63;
}
// the integer path takes boxes of up to 1000 cells per axis with 1/4 <= d < 8
// and 0 < h_min, h_c < 8 (lattice units); everything else runs the FP64 body.
// Positions are exact in units of 2^-54 (2^-53 from 512 cells on) except
// below one cell from the origin, where they lose half an FP64 rounding of a
// separation of one cell.
__host__ __device__ inline FxBox fx_box(const int n[3], double dmin, double dmax, double h_c, double h_min, double mu) {
    FxBox b;
    std::memset(&b, 0, sizeof b);
    b.ok = n[0] <= 1000 && n[1] <= 1000 && n[2] <= 1000 && dmin >= 0.25 && dmax < 8.0 && h_c >= 0.0 && h_c < 8.0 &&
           h_min > 0x1p-40 && h_min < 8.0 && mu > 0x1p-100 && mu < 0x1p100;
    if (!b.ok) return b;
    b.frac = n[0] < 512 && n[1] < 512 && n[2] < 512 ? 54 : 53;
    b.hc = fx_from_pos(h_c, 56);
    b.hmin = fx_from_pos(h_min, 56);
    fx_split(h_min, b.hmin_m, b.hmin_e);
    fx_split(1.57079632679489661923 * mu, b.c_m, b.c_e);
    return b;
}

// v >= 0 truncated to single precision, relative error below 2^-20
__host__ __device__ __forceinline__ float fx_approx(double v) {
    const u32 hi = (u32)(fx_bits(v) >> 32);
    const int e = (int)(hi >> 20) - 1023 + 127;
    const u32 f = e <= 0 ? 0u : (e >= 255 ? 0x7f800000u : ((u32)e << 23) | ((hi & 0xfffffu) << 3));
#ifdef __CUDA_ARCH__
    return __uint_as_float(f);
#else
    float r;
    std::memcpy(&r, &f, 4);
    return r;
#endif
}

enum : int { FX_NONE = 0, FX_LUB = 1, FX_EXACT = 2 };

struct FxPair {
    double n[3];         // unit normal from i to j
    double alpha, beta;  // shear and squeeze coefficients a_sh (2/(h+<d>))^2 and a_sq, before the limiter
};

// The lubrication coefficients (Sec. 3.1.3) at the floored gap hh = Hm 2^He (leading
// bit of Hm set) and 1/<d> = I 2^-59: alpha and beta as in FxPair.  FX_LUB, FX_NONE (both
// are zero) or FX_EXACT (out of range).
__host__ __device__ __forceinline__ int fx_lub(u64 Hm, int He, u64 I, const FxBox &bx, double &alpha, double &beta) {
    // ir = hh/<d>, P = hh/<d>^2
    const int li = fx_clz(I);
    const u64 Im = I << li;
    u64 ir = fx_mulhi(Hm, Im);
    int ire = He + 5 - li;  // (+64 - 59)
    const int l1 = (ir >> 63) ? 0 : 1;
    ir <<= l1;
    ire -= l1;
    if (ire >= -63) return FX_NONE;  // hh >= <d>: both coefficients are negative, clamped to zero
    const int q = -64 - ire;         // ir = ir_m 2^-64 2^-q
    if (q > 28) return FX_EXACT;
    u64 P = fx_mulhi(ir, Im);
    int Pe = ire + 5 - li;
    const int l2 = (P >> 63) ? 0 : 1;
    P <<= l2;
    Pe -= l2;
    // 1/P: y (1 + e + e^2), P = p 2^(64+Pe), p in [1/2, 1)
    u32 V = (u32)(fx_rcp_seed((float)(u32)(P >> 32) * 0x1p-32f) * 0x1p30f);
    V = V > 0x7fffffffu ? 0x7fffffffu : V;
    const i64 e1 = (i64)((1ull << 63) - fx_mulhi(P, (u64)V << 33));  // 2^-63
    const i64 f1 = (i64)(int)(e1 >> 12);
    const i64 c1 = e1 + ((f1 * f1) >> 39);
    const u64 RP = ((u64)V << 32) + (u64)(((c1 >> 32) * (i64)V) * 2) + (((u64)(u32)c1 * V) >> 31);  // 2^-62, in (1, 2]
    // L = ln(<d>/2hh) = -ln(2 ir), 2 ir = m 2^-q, m = ir_m 2^-63 in [1, 2)
#ifdef __CUDA_ARCH__
    const FxLogRow row = fx_log_dev[(int)(ir >> 56) & 127];
#else
    const FxLogRow row = fx_log_host[(int)(ir >> 56) & 127];
#endif
    const i64 u = (i64)(fx_mulhi(ir, (u64)row.C << 47)) - (i64)(1ull << 62);  // 2^-62, |u| < 2^-7.9
    const int v = (int)(u >> 24);                                             // 2^-38
    const int t6 = 357913941 - (fx_mulhi32(v, 306783378) >> 6);               // 2^-31: 1/6 - u/7
    const int t5 = 429496730 - (fx_mulhi32(v, t6) >> 6);                      // 1/5 - u t6
    const int t4 = 536870912 - (fx_mulhi32(v, t5) >> 6);                      // 1/4 - u t5
    const i64 T3 = 1537228672809129301ll - (((i64)v * t4) >> 7);  // 2^-62: 1/3 - u t4
    const i64 T2 = (i64)(1ull << 61) - (fx_mulhi_s(u, T3) << 2);       // 2^-62: 1/2 - u T3
    const i64 u2 = fx_mulhi_s(u, u);                                   // 2^-60
    const i64 ln1p = (u >> 4) - fx_mulhi_s(u2, T2);                    // 2^-58
    const i64 L = (i64)q * DPS_FX_LN2_Q58 - row.T - ln1p;              // 2^-58
    // a_sh (2/(h+<d>))^2 = (pi/2) mu <d> L = c (L ir)/P and a_sq = (pi/2) mu
    // <d> 3 (r/4 + 18/40 L + 9/84 L ir) = c (3/4 + L ir (27/20 + 9/28 ir))/P
    const u64 CP = fx_mulhi(RP, bx.c_m);  // c/P = CP 2^(c_e-Pe-62)
    const u64 La = (u64)(L < 0 ? -L : L);
    const int lL = fx_clz(La | 1);
    const u64 LI = fx_mulhi(La << lL, ir);  // |L| ir = LI 2^-(58+lL+q)
    alpha = L > 0 ? fx_to_double(fx_mulhi(LI, CP), 56 + lL + q + Pe - bx.c_e) : 0.0;
    const int st = lL + q - 2;  // >= 3: |L| ir < 1
    const i64 ta = (i64)(LI >> (st > 63 ? 63 : st));  // 2^-60
    const i64 W = 6225776124876973670ll + (i64)fx_mulhi(ir >> q, 1482327648780231826ull);  // 27/20 + 9/28 ir, 2^-62
    const i64 B3 = (3ll << 56) + fx_mulhi_s(L < 0 ? -ta : ta, W);  // 2^-58
    beta = B3 > 0 ? fx_to_double(fx_mulhi((u64)B3 << 4, CP), 60 + Pe - bx.c_e) : 0.0;
    return FX_LUB;
}

// One pair (Sec. 3.1.3).  dx: x_j - x_i (minimum image) in units of 2^-frac, S
// = rad_i + rad_j (fx_radius), I = fx_inv_d of i plus that of j.  FX_EXACT:
// the pair overlaps or leaves the range of this path, the FP64 body decides;
// FX_NONE: no force; FX_LUB: o holds the coefficients.
__host__ __device__ __forceinline__ int fx_pair(const i64 dx[3], i64 S, u64 I, const FxBox &bx, FxPair &o) {
    u64 a[3];
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int k = 0; k < 3; ++k) a[k] = (u64)(dx[k] < 0 ? -dx[k] : dx[k]);
    // leading bit of the largest component at bit 62: a = x' 2^63, |x'| < 1
    const u64 any = a[0] | a[1] | a[2];
    const int s = fx_clz(any) - 1;
    const int gf = s + bx.frac - 3, sl = gf - 56;
    if (sl < 0 || sl > 24) return FX_EXACT;  // |dx| >= 16, or far below any radius of the path
    u64 X[3], N2 = 0;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int k = 0; k < 3; ++k) {
        X[k] = a[k] << s;
        N2 += fx_mulhi(X[k], X[k]);  // |x'|^2 in units of 2^-62, in [1/4, 3)
    }
    // r = 1/|x'|: y (1 + e/2 + 3/8 e^2) with e = 1 - |x'|^2 y^2
    const float yf = fx_rsqrt_seed((float)(u32)(N2 >> 32) * 0x1p-30f);
    const u32 Y = (u32)(yf * 0x1p30f);
    const i64 e = (i64)(1ull << 58) - (i64)fx_mulhi(N2, (u64)Y * Y);  // 2^-58
    const i64 eh = (i64)(int)(e >> 8);
    const i64 c = (e >> 1) + ((3 * ((eh * eh) >> 42)) >> 3);
    const u64 R = ((u64)Y << 32) + (u64)(((c >> 32) * (i64)Y) * 64) + (((u64)(u32)c * Y) >> 26);  // 2^-62
    // gap in units of 2^-gf: |dx| - S
    const i64 D = (i64)fx_mulhi(N2, R);
    if ((S >> (62 - sl)) != 0) return FX_EXACT;  // S past the scale of |dx|: deep overlap
    const i64 G = D - (S << sl);
    if (G < 0) return FX_EXACT;
    if ((G >> sl) >= bx.hc) return FX_NONE;
    // the floored gap hh = Hm 2^He
    u64 Hm = bx.hmin_m;
    int He = bx.hmin_e;
    if ((G >> sl) >= bx.hmin) {
        const int lz = fx_clz((u64)G);
        Hm = (u64)G << lz;
        He = -gf - lz;
    }
    const int kind = fx_lub(Hm, He, I, bx, o.alpha, o.beta);
    if (kind != FX_LUB) return kind;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
    for (int k = 0; k < 3; ++k) {
        o.n[k] = fx_with_sign(fx_to_double(fx_mulhi(X[k], R), 61), dx[k]);
    }
    return FX_LUB;
}

// A wall of gap h >= 0 (FP64: one subtraction, exact for small gaps; through the
// positions' fixed-point copies the gap 1e-5 of a sphere at x < 1/4 would lose five
// digits) and I = fx_inv_d of the sphere, 1/<d> = 1/(2 d).
__host__ __device__ __forceinline__ int fx_wall(double h, u64 I, double h_c, double h_min, const FxBox &bx,
                                                double &alpha, double &beta) {
    if ((i64)fx_bits(h) < 0) return FX_EXACT;  // overlap
    if (fx_bits(h) >= fx_bits(h_c)) return FX_NONE;
    u64 Hm = bx.hmin_m;
    int He = bx.hmin_e;
    if (fx_bits(h) >= fx_bits(h_min)) fx_split(h, Hm, He);
    return fx_lub(Hm, He, I, bx, alpha, beta);
}

}  // namespace dps
