// lbm.cu -- GNS lattice Boltzmann kernels (Sec. 3.2.2, Eqs. LBM_Equation,
// LBM_EQ, Forcing, MacVel) and the per-step fluid fields of Sec. 3.2.3.
//
// K1 collide-stream: one fused pass, in place with the AA pattern.  Even
//    parity reads and writes only the own cell (the post-collision value of
//    direction q goes to plane opp(q)); odd parity reads the upstream values
//    and writes the downstream cells.  Halfway bounce-back at wall faces is
//    folded into the odd-parity index map.  HBM traffic per cell: 19 loads and
//    19 stores of the PDF type plus eps_f and f_pf (4 loads of the field type).
//    FP64: 207 FP64 warp instructions of ~19 cycles per 32 cells bound this
//    pass; it runs in 64-bit fixed point (lbm_fx.cuh), ~1500 integer
//    instructions of which two to four issue per cycle.  128^3, walls at z:
//    815 -> 215 us; 256^3, coupled step: 4.88 -> 1.67 ms (floor at the
//    measured copy rate: 0.10 and 0.83 ms).  With a
//    per-cell tau_e only tau_e is FP64: 75 x 61 x 90, 229 -> 105 us.
// K2a moments: rho, j of f(x,t), u_D = (j + f_ext/2)/(rho eps_f) and
//    1/(rho eps_f); one PDF read.
// K2b fields: stencil over rho and u_D giving grad(eps_f p) and Du_f/Dt.
#include "box.cuh"
#include "lbm_dev.cuh"
#include "lbm_fx.cuh"

namespace dps {

// Eq. tau_e for one cell: tau_* from the Eilers viscosity of eps_p = 1 - eps_f
// (Eq. visc_eilers; eps_p/eps_cp capped at 0.9 where it diverges) plus the
// Smagorinsky tau_t (Eqs. visc_turb, tau_t) from the non-equilibrium momentum
// flux Q_ab = sum_q c_a c_b (f_q - f_q^eq) = Pi_ab - c_s^2 rho delta_ab -
// rho u_a u_b / eps.  Qbar = sqrt(2 sum Q_ab Q_ab); tau_t solves
// tau_t (tau_* + tau_t) = C_S^2 Qbar / (2 rho c_s^4) and is taken in the
// cancellation-free form x / (2 (sqrt(tau_*^2 + x) + tau_*)).  With DEV the
// second moments are of the deviations: Pi~_ab = Pi_ab - c_s^2 delta_ab, and
// s = rho - 1.
template <typename CT, bool DEV>
__device__ __forceinline__ CT tau_cell(const CT f[Q], CT s, CT rho, CT ux, CT uy, CT uz, CT e, CT ie, CT tau,
                                       int eilers, int smag) {
    CT ts = tau;
    if (eilers) {
        CT r = (CT(1) - e) * CT(1.0 / 0.64);
        r = r < CT(0) ? CT(0) : (r > CT(0.9) ? CT(0.9) : r);
        const CT a = CT(1) + CT(1.25 * 0.64) * r / (CT(1) - r);
        ts = CT(0.5) + (tau - CT(0.5)) * (a * a);
    }
    if (!smag) return ts;
    CT P[6] = {0, 0, 0, 0, 0, 0};  // xx yy zz xy xz yz
#pragma unroll
    for (int k = 1; k <= 9; ++k) {
        const CT p = f[k] + f[k + 9];
        if (CX(k) != 0) P[0] += p;
        if (CY(k) != 0) P[1] += p;
        if (CZ(k) != 0) P[2] += p;
        if (CX(k) * CY(k) != 0) P[3] += CT(CX(k) * CY(k)) * p;
        if (CX(k) * CZ(k) != 0) P[4] += CT(CX(k) * CZ(k)) * p;
        if (CY(k) * CZ(k) != 0) P[5] += CT(CY(k) * CZ(k)) * p;
    }
    const CT iso = CT(1.0 / 3.0) * (DEV ? s : rho);
    const CT ri = rho * ie;
    const CT qxx = P[0] - iso - ri * ux * ux, qyy = P[1] - iso - ri * uy * uy, qzz = P[2] - iso - ri * uz * uz;
    const CT qxy = P[3] - ri * ux * uy, qxz = P[4] - ri * ux * uz, qyz = P[5] - ri * uy * uz;
    const CT q2 = qxx * qxx + qyy * qyy + qzz * qzz + CT(2) * (qxy * qxy + qxz * qxz + qyz * qyz);
    const CT x = CT(2 * 0.01 * 9) * m_sqrt(CT(2) * q2) / rho;  // 2 C_S^2 Qbar / (rho c_s^4)
    return ts + x / (CT(2) * (m_sqrt(ts * ts + x) + ts));
}

// K1 body for one cell: load the 19 populations (AA parity PAR), relax them
// (Eq. LBM_Equation, relax_cell) and store each opposite pair as soon as it
// is computed, which keeps few values live.  VISC: the box may
// relax with a per-cell tau_e (vmode bit 0 Eilers, bit 1 Smagorinsky).
template <typename ST, typename FT, typename CT, int PAR, bool VISC>
__device__ __forceinline__ void relax_store_cell(ST *__restrict__ pdf, CT f[Q], const NbDelta &D, bool in,
                                                 const Geom &g, CT e, CT fpx, CT fpy, CT fpz, long long N, long long c,
                                                 CT fbx, CT fby, CT fbz, CT omega_box, CT kf_box, CT tau, int vmode,
                                                 int *status, const FxFluid *ff = nullptr);

template <typename ST, typename FT, typename CT, int PAR, bool VISC>
__device__ __forceinline__ void collide_stream_cell(ST *__restrict__ pdf, const FT *__restrict__ eps,
                                                    const FT *__restrict__ fpf, const Geom &g, long long c, CT fbx,
                                                    CT fby, CT fbz, CT omega_box, CT kf_box, CT tau, int vmode,
                                                    int *status, const FxFluid *ff = nullptr) {
    const long long N = g.ncell;
    NbDelta D;
    bool in = false;
    CT f[Q];
    if (PAR) {
        int ix, iy, iz;
        cell_coords(g, c, ix, iy, iz);
        D = neighbour_deltas(g, ix, iy, iz);
        in = no_wall_neighbour(D);
        if (in)
            load_pdfs_wall_free<ST, CT>(pdf, (unsigned)N, (unsigned)c, D, f);
        else
            load_pdfs<ST, CT, PAR>(pdf, N, c, D, f);
    } else {
        load_pdfs<ST, CT, PAR>(pdf, N, c, D, f);
    }
    relax_store_cell<ST, FT, CT, PAR, VISC>(pdf, f, D, in, g, (CT)eps[c], (CT)fpf[c], (CT)fpf[N + c],
                                                   (CT)fpf[2 * N + c], N, c, fbx, fby, fbz, omega_box, kf_box, tau,
                                                   vmode, status, ff);
}

// two cells per thread (c and c + stride): the loads of both are issued before
// either is relaxed, which doubles the bytes in flight per warp
template <typename ST, typename FT, typename CT, int PAR, bool VISC>
__device__ __forceinline__ void collide_stream_cell2(ST *__restrict__ pdf, const FT *__restrict__ eps,
                                                     const FT *__restrict__ fpf, const Geom &g, long long c,
                                                     long long c2, bool two, CT fbx, CT fby, CT fbz, CT omega_box,
                                                     CT kf_box, CT tau, int vmode, int *status) {
    const long long N = g.ncell;
    NbDelta D, D2;
    bool in = false, in2 = false;
    CT f[Q], f2[Q];
    if (PAR) {
        int ix, iy, iz;
        cell_coords(g, c, ix, iy, iz);
        D = neighbour_deltas(g, ix, iy, iz);
        in = no_wall_neighbour(D);
        if (in)
            load_pdfs_wall_free<ST, CT>(pdf, (unsigned)N, (unsigned)c, D, f);
        else
            load_pdfs<ST, CT, PAR>(pdf, N, c, D, f);
        if (two) {
            cell_coords(g, c2, ix, iy, iz);
            D2 = neighbour_deltas(g, ix, iy, iz);
            in2 = no_wall_neighbour(D2);
            if (in2)
                load_pdfs_wall_free<ST, CT>(pdf, (unsigned)N, (unsigned)c2, D2, f2);
            else
                load_pdfs<ST, CT, PAR>(pdf, N, c2, D2, f2);
        }
    } else {
        load_pdfs<ST, CT, PAR>(pdf, N, c, D, f);
        if (two) load_pdfs<ST, CT, PAR>(pdf, N, c2, D2, f2);
    }
    const CT e = (CT)eps[c], e2 = two ? (CT)eps[c2] : CT(1);
    const CT a0 = (CT)fpf[c], a1 = (CT)fpf[N + c], a2 = (CT)fpf[2 * N + c];
    CT b0 = 0, b1 = 0, b2 = 0;
    if (two) {
        b0 = (CT)fpf[c2];
        b1 = (CT)fpf[N + c2];
        b2 = (CT)fpf[2 * N + c2];
    }
    relax_store_cell<ST, FT, CT, PAR, VISC>(pdf, f, D, in, g, e, a0, a1, a2, N, c, fbx, fby, fbz, omega_box,
                                                   kf_box, tau, vmode, status);
    if (two)
        relax_store_cell<ST, FT, CT, PAR, VISC>(pdf, f2, D2, in2, g, e2, b0, b1, b2, N, c2, fbx, fby, fbz,
                                                       omega_box, kf_box, tau, vmode, status);
}

// two-element vectors of the stored type (low-precision forms): float2 or
// half2, converted exactly to and from the FP32 arithmetic (the FP16 stores
// round each element to nearest even, as the scalar stores do)
template <typename ST> struct Vec2;
template <> struct Vec2<float> {
    __device__ static inline void load(const float *p, float &a, float &b) {
        const float2 v = *reinterpret_cast<const float2 *>(p);
        a = v.x;
        b = v.y;
    }
    __device__ static inline void store(float *p, float a, float b) { *reinterpret_cast<float2 *>(p) = make_float2(a, b); }
};
template <> struct Vec2<double> {  // for completeness: the FP64 form keeps the scalar variant
    __device__ static inline void load(const double *p, double &a, double &b) {
        const double2 v = *reinterpret_cast<const double2 *>(p);
        a = v.x;
        b = v.y;
    }
    __device__ static inline void store(double *p, double a, double b) {
        *reinterpret_cast<double2 *>(p) = make_double2(a, b);
    }
};
template <> struct Vec2<__half> {
    __device__ static inline void load(const __half *p, float &a, float &b) {
        const float2 v = __half22float2(*reinterpret_cast<const __half2 *>(p));
        a = v.x;
        b = v.y;
    }
    __device__ static inline void store(__half *p, float a, float b) {
        *reinterpret_cast<__half2 *>(p) = __floats2half2_rn(a, b);
    }
};

template <typename ST, typename CT, bool VISC>
__device__ __forceinline__ void relax_cell(CT f[Q], CT e, CT fpx, CT fpy, CT fpz, CT fbx, CT fby, CT fbz,
                                           CT omega_box, CT kf_box, CT tau, int vmode, bool flag, int *status);

// the populations of the cells c and c + 1 (without a wall neighbour at odd parity)
template <typename ST, typename CT, int PAR>
__device__ __forceinline__ void load_pair(const ST *__restrict__ pdf, unsigned Nu, unsigned cu, const NbDelta &D,
                                          const NbDelta &D1, CT f[Q], CT f1[Q]) {
    Vec2<ST>::load(pdf + cu, f[0], f1[0]);
#pragma unroll
    for (int q = 1; q < Q; ++q) {
        if (PAR == 0) {
            Vec2<ST>::load(pdf + ((unsigned)q * Nu + cu), f[q], f1[q]);
        } else if (CX(q) == 0) {
            Vec2<ST>::load(pdf + ((unsigned)OPP(q) * Nu + cu + wall_free_delta(D, 0, -CY(q), -CZ(q))), f[q], f1[q]);
        } else {
            f[q] = Store<ST>::load(pdf + ((unsigned)OPP(q) * Nu + cu + wall_free_delta(D, -CX(q), -CY(q), -CZ(q))));
            f1[q] = Store<ST>::load(pdf + ((unsigned)OPP(q) * Nu + cu + 1u +
                                           wall_free_delta(D1, -CX(q), -CY(q), -CZ(q))));
        }
    }
}

// two consecutive cells c, c+1 (c and ncell even).  Even parity: own-cell
// accesses only, any pair.  Odd parity: two cells of one x row (nx even: the
// plane offsets, the pair and every y / z neighbour offset are even), both
// without a wall neighbour.  A population whose memory offset keeps the pair aligned (even
// parity: every one; odd parity: those with c_x = 0) moves as one
// two-element vector, half the load and store instructions of the scalar
// path; the x-moving populations of the odd parity stay scalar.  A pair next
// to a wall takes the scalar path cell by cell.  The relaxation is that of
// the scalar path, so the results are the same bits.
template <typename ST, typename FT, typename CT, int PAR, bool VISC>
__device__ __forceinline__ void collide_stream_vec2(ST *__restrict__ pdf, const FT *__restrict__ eps,
                                                    const FT *__restrict__ fpf, const Geom &g, long long c, CT fbx,
                                                    CT fby, CT fbz, CT omega_box, CT kf_box, CT tau, int vmode,
                                                    int *status) {
    const long long N = g.ncell;
    NbDelta D, D1;
    if (PAR) {
        int ix, iy, iz;
        cell_coords(g, c, ix, iy, iz);
        D = neighbour_deltas(g, ix, iy, iz);
        D1 = neighbour_deltas(g, ix + 1, iy, iz);
    }
    if (PAR && (!no_wall_neighbour(D) || !no_wall_neighbour(D1))) {
        collide_stream_cell<ST, FT, CT, PAR, VISC>(pdf, eps, fpf, g, c, fbx, fby, fbz,
                                                          omega_box, kf_box, tau, vmode, status);
        collide_stream_cell<ST, FT, CT, PAR, VISC>(pdf, eps, fpf, g, c + 1, fbx, fby, fbz,
                                                          omega_box, kf_box, tau, vmode, status);
        return;
    }
    const unsigned Nu = (unsigned)N, cu = (unsigned)c;
    CT f[Q], f1[Q];
    load_pair<ST, CT, PAR>(pdf, Nu, cu, D, D1, f, f1);
    // eps_f and f_pf of the pair as two-element vectors too (FT is float
    // in the forms that take this path; c and N are even)
    CT e0, e1, a[3], b[3];
    Vec2<FT>::load(eps + cu, e0, e1);
#pragma unroll
    for (int k = 0; k < 3; ++k) Vec2<FT>::load(fpf + ((unsigned)k * Nu + cu), a[k], b[k]);
    relax_cell<ST, CT, VISC>(f, e0, a[0], a[1], a[2], fbx, fby, fbz, omega_box, kf_box, tau, vmode, true,
                                    status);
    relax_cell<ST, CT, VISC>(f1, e1, b[0], b[1], b[2], fbx, fby, fbz, omega_box, kf_box, tau, vmode, true,
                                    status);
    Vec2<ST>::store(pdf + cu, f[0], f1[0]);
#pragma unroll
    for (int k = 1; k <= 9; ++k) {
        if (PAR == 0) {
            Vec2<ST>::store(pdf + ((unsigned)(k + 9) * Nu + cu), f[k], f1[k]);
            Vec2<ST>::store(pdf + ((unsigned)k * Nu + cu), f[k + 9], f1[k + 9]);
        } else if (CX(k) == 0) {
            // (the offsets are summed in 32-bit unsigned arithmetic, where a
            // negative neighbour delta wraps, before they move the pointer)
            Vec2<ST>::store(pdf + ((unsigned)k * Nu + cu + wall_free_delta(D, 0, CY(k), CZ(k))), f[k], f1[k]);
            Vec2<ST>::store(pdf + ((unsigned)(k + 9) * Nu + cu + wall_free_delta(D, 0, -CY(k), -CZ(k))), f[k + 9],
                            f1[k + 9]);
        } else {
            store_pair_wall_free<ST, CT>(pdf, Nu, cu, D, k, f[k], f[k + 9]);
            store_pair_wall_free<ST, CT>(pdf, Nu, cu + 1u, D1, k, f1[k], f1[k + 9]);
        }
    }
}

// Correctly rounded single operations: the relaxation below spells out every
// multiply, add and fused multiply-add, so each K1 variant (register budget,
// cells per thread) rounds exactly alike and a box's result does not depend on
// the launch shape the autotuner picks.
__device__ __forceinline__ float r_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double r_fma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float r_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double r_mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float r_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double r_add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float r_sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double r_sub(double a, double b) { return __dsub_rn(a, b); }

// relaxation (Eq. LBM_Equation) of one cell whose populations f, eps_f and
// f_pf are loaded: BGK relaxation towards the porous equilibrium (Eq.
// LBM_EQ) plus the Guo forcing term (Eq. Forcing); f is overwritten with the
// post-collision populations.  With deviation storage (shifted forms) the
// populations are f_q - w_q (rho_0 = 1): rho = 1 + sum, and the update of a
// deviation is f' - w = (1-omega)(f - w) + omega(f^eq - w) + F.  The update
// is written per opposite pair (q, q+9): the even part in c of
// omega f^eq + F is E = K0 + cu (K1 cu + K2 cF), the odd part
// O = K3 cu + K4 cF, with K0..K4 fixed per weight class.
// `flag`: report a non-finite or non-positive density.
template <typename ST, typename CT, bool VISC>
__device__ __forceinline__ void relax_cell(CT f[Q], CT e, CT fpx, CT fpy, CT fpz, CT fbx, CT fby, CT fbz,
                                           CT omega_box, CT kf_box, CT tau, int vmode, bool flag, int *status) {
    constexpr bool DEV = Store<ST>::shifted;
    // f_ext = f_pf + eps_f f_b (Eq. Forcing)
    const CT Fx = r_fma(e, fbx, fpx);
    const CT Fy = r_fma(e, fby, fpy);
    const CT Fz = r_fma(e, fbz, fpz);
    CT s = f[0], jx = 0, jy = 0, jz = 0;
#pragma unroll
    for (int k = 1; k <= 9; ++k) {
        s = r_add(s, r_add(f[k], f[k + 9]));
        const CT d = r_sub(f[k], f[k + 9]);
        if (CX(k) != 0) jx = CX(k) > 0 ? r_add(jx, d) : r_sub(jx, d);
        if (CY(k) != 0) jy = CY(k) > 0 ? r_add(jy, d) : r_sub(jy, d);
        if (CZ(k) != 0) jz = CZ(k) > 0 ? r_add(jz, d) : r_sub(jz, d);
    }
    const CT rho = DEV ? r_add(CT(1), s) : s;
    if (flag && (!(rho > CT(0)) || !(rho < CT(1e30)))) atomicOr(status, ST_NAN);
    // 1/rho and 1/eps_f from one division (the FP64 form is bound by its
    // FP64 instruction count)
    const CT t = CT(1) / r_mul(rho, e);
    const CT ir = r_mul(e, t), ie = r_mul(rho, t);
    const CT ux = r_mul(r_fma(CT(0.5), Fx, jx), ir);  // Eq. MacVel
    const CT uy = r_mul(r_fma(CT(0.5), Fy, jy), ir);
    const CT uz = r_mul(r_fma(CT(0.5), Fz, jz), ir);
    CT omega = omega_box, kf = kf_box;
    if (VISC && vmode) {
        omega = CT(1) / tau_cell<CT, DEV>(f, s, rho, ux, uy, uz, e, ie, tau, vmode & 1, vmode & 2);
        kf = r_fma(CT(-0.5), omega, CT(1));
    }
    const CT uu = r_fma(ux, ux, r_fma(uy, uy, r_mul(uz, uz)));
    const CT uF = r_fma(ux, Fx, r_fma(uy, Fy, r_mul(uz, Fz)));
    const CT om1 = r_sub(CT(1), omega);
    const CT b2 = r_mul(r_mul(CT(-1.5), uu), ie);
    const CT e0 = DEV ? r_mul(omega, r_fma(rho, b2, s)) : r_mul(r_mul(omega, rho), r_add(CT(1), b2));
    const CT f0 = r_mul(r_mul(r_mul(CT(-3), kf), uF), ie);
    const CT ef = r_add(e0, f0);
    const CT k1 = r_mul(r_mul(r_mul(omega, rho), CT(4.5)), ie), k2 = r_mul(r_mul(CT(9), kf), ie);
    const CT k3 = r_mul(r_mul(CT(3), omega), rho), k4 = r_mul(CT(3), kf);
    f[0] = r_fma(om1, f[0], r_mul((CT)WQ(0), ef));
#pragma unroll
    for (int k = 1; k <= 9; ++k) {
        const CT w = (CT)WQ(k);
        CT cu = 0, cF = 0;
        if (CX(k) != 0) { cu = CX(k) > 0 ? r_add(cu, ux) : r_sub(cu, ux); cF = CX(k) > 0 ? r_add(cF, Fx) : r_sub(cF, Fx); }
        if (CY(k) != 0) { cu = CY(k) > 0 ? r_add(cu, uy) : r_sub(cu, uy); cF = CY(k) > 0 ? r_add(cF, Fy) : r_sub(cF, Fy); }
        if (CZ(k) != 0) { cu = CZ(k) > 0 ? r_add(cu, uz) : r_sub(cu, uz); cF = CZ(k) > 0 ? r_add(cF, Fz) : r_sub(cF, Fz); }
        const CT E = r_mul(w, r_fma(cu, r_fma(k1, cu, r_mul(k2, cF)), ef));
        const CT O = r_mul(w, r_fma(k3, cu, r_mul(k4, cF)));
        const CT vk = r_fma(om1, f[k], r_add(E, O)), vo = r_fma(om1, f[k + 9], r_sub(E, O));
        f[k] = vk;
        f[k + 9] = vo;
    }
}

// relaxation and parity-aware stores of one cell
template <typename ST, typename FT, typename CT, int PAR, bool VISC>
__device__ __forceinline__ void relax_store_cell(ST *__restrict__ pdf, CT f[Q], const NbDelta &D, bool in,
                                                 const Geom &g, CT e, CT fpx, CT fpy, CT fpz, long long N, long long c,
                                                 CT fbx, CT fby, CT fbz, CT omega_box, CT kf_box, CT tau, int vmode,
                                                 int *status, const FxFluid *ff) {
    bool done = false;
    if constexpr (sizeof(ST) == 8) {
        u64 b[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) b[q] = fx_bits(f[q]);
        done = fx_relax<VISC>(b, e, fpx, fpy, fpz, *ff, tau, vmode, f);
    }
    if (!done)
        relax_cell<ST, CT, VISC>(f, e, fpx, fpy, fpz, fbx, fby, fbz, omega_box, kf_box, tau, vmode, true, status);
    Store<ST>::store(pdf + (unsigned)c, f[0]);
#pragma unroll
    for (int k = 1; k <= 9; ++k) {
        if (PAR && in)
            store_pair_wall_free<ST, CT>(pdf, (unsigned)N, (unsigned)c, D, k, f[k], f[k + 9]);
        else
            store_pair<ST, CT, PAR>(pdf, N, c, D, k, f[k], f[k + 9]);
    }
}

template <typename CT> __device__ __forceinline__ CT pick(double d, float f);
template <> __device__ __forceinline__ double pick<double>(double d, float) { return d; }
template <> __device__ __forceinline__ float pick<float>(double, float f) { return f; }

#ifndef DPS_K1_MINB
#define DPS_K1_MINB 3  // FP64: 128-thread blocks per SM the register budget is sized for
#endif
#ifndef DPS_K1V_MINB
#define DPS_K1V_MINB 3  // the same with a per-cell tau_e
#endif
// K1: every cell tile of every box, AA parity PAR (common to the batch).
template <typename ST, typename FT, typename CT, int PAR, int MINB, bool VISC, int CPT>
__global__ void __launch_bounds__(128, MINB) k_collide_stream(const BoxDev *__restrict__ boxes,
                                                           const Tile *__restrict__ tiles, int ntiles) {
    DPS_FOR_TILES(tiles, ntiles, t) {
        const Tile tl = tiles[t];
        const BoxDev &B = boxes[tl.box];
        const Geom g = B.g;
        ST *pdf = (ST *)B.pdf;
        const FT *eps = (const FT *)B.eps, *fpf = (const FT *)B.fpf;
        const CT fbx = pick<CT>(B.ph.fb[0], B.ph.fb_f[0]), fby = pick<CT>(B.ph.fb[1], B.ph.fb_f[1]),
                 fbz = pick<CT>(B.ph.fb[2], B.ph.fb_f[2]);
        const CT omega = pick<CT>(B.ph.omega, B.ph.omega_f), kf = pick<CT>(B.ph.kf, B.ph.kf_f);
        const CT tau = (CT)B.ph.tau;
        const int vmode = VISC ? (B.ph.eilers ? 1 : 0) | (B.ph.smag ? 2 : 0) : 0;
        int *st = B.status;
        if (CPT == 3 && sizeof(ST) < 8 && !(g.ncell & 1) && !((tl.begin | tl.end) & 1) &&
            (!PAR || !(g.n[0] & 1))) {
            // vector pairs; the odd parity at odd nx moves scalars, two cells a
            // thread in FP16 (161 x 150 x 139: 131 -> 107 us a step), one in
            // FP32 (two: 148 us against 135)
            for (long long c = tl.begin + 2 * threadIdx.x; c < tl.end; c += 2 * blockDim.x)
                collide_stream_vec2<ST, FT, CT, PAR, VISC>(pdf, eps, fpf, g, c, fbx, fby, fbz, omega, kf, tau, vmode,
                                                           st);
        } else if (CPT == 1 || (CPT == 3 && sizeof(ST) == 4)) {
            for (long long c = tl.begin + threadIdx.x; c < tl.end; c += blockDim.x)
                collide_stream_cell<ST, FT, CT, PAR, VISC>(pdf, eps, fpf, g, c, fbx, fby, fbz,
                                                                  omega, kf, tau, vmode, st, &B.ph.ff);
        } else {
            for (long long c = tl.begin + threadIdx.x; c < tl.end; c += 2 * blockDim.x) {
                const long long c2 = c + blockDim.x;
                collide_stream_cell2<ST, FT, CT, PAR, VISC>(pdf, eps, fpf, g, c, c2, c2 < tl.end,
                                                                   fbx, fby, fbz, omega, kf, tau, vmode, st);
            }
        }
    }
}

// K2a body: rho, j and u_D = (j + f_ext/2)/(rho eps) with the applied f_ext.
// o: rho, j (3), 1/(rho eps), u_D (3)
template <typename ST, typename CT>
__device__ __forceinline__ void moments_of(const CT f[Q], CT e, CT fp0, CT fp1, CT fp2, CT fbx, CT fby, CT fbz,
                                           CT o[8]) {
    CT rho, jx, jy, jz, s = 0;
    bool exact = false;
    if constexpr (sizeof(ST) == 8) {
        // the sums are exact in units of 2^-62 (FP64: 57 FP64 instructions a
        // cell, here 9); 1/(rho eps) by Newton's iteration on integers
        u64 b[Q];
        i64 fi[Q], r, j[3];
#pragma unroll
        for (int q = 0; q < Q; ++q) b[q] = fx_bits(f[q]);
        if (fx_populations(b, fi, r, j) && r > (1ll << 61) && e > 0.125 && e <= 1.0) {
            int lz;
            const u64 R = fx_recip(r, fx_from_pos(e, 62), lz);
            s = fx_to_double(R, 64 - lz);
            rho = fx_to_double((u64)r, 62);
            jx = fx_signed_to_double(j[0], 62);
            jy = fx_signed_to_double(j[1], 62);
            jz = fx_signed_to_double(j[2], 62);
            exact = true;
        }
    }
    if (!exact) {
        moments(f, rho, jx, jy, jz);
        if (Store<ST>::shifted) rho += CT(1);  // deviations: sum of the shifts w_q is 1
        s = CT(1) / (rho * e);
    }
    const CT Fx = fp0 + e * fbx, Fy = fp1 + e * fby, Fz = fp2 + e * fbz;
    o[0] = rho;
    o[1] = jx;
    o[2] = jy;
    o[3] = jz;
    o[4] = s;  // the first subcycle's drag interpolation reuses it
    o[5] = (jx + CT(0.5) * Fx) * s;
    o[6] = (jy + CT(0.5) * Fy) * s;
    o[7] = (jz + CT(0.5) * Fz) * s;
}

template <typename ST, typename FT, typename CT, int PAR>
__device__ __forceinline__ void moments_cell(const ST *__restrict__ pdf, const FT *__restrict__ eps,
                                             const FT *__restrict__ fpf, const Geom &g, long long c, CT fbx, CT fby,
                                             CT fbz, FT *__restrict__ rho_o, FT *__restrict__ j_o,
                                             FT *__restrict__ uD, FT *__restrict__ ire) {
    const long long N = g.ncell;
    int ix, iy, iz;
    cell_coords(g, c, ix, iy, iz);
    NbDelta D = neighbour_deltas(g, ix, iy, iz);
    CT f[Q], o[8];
    load_pdfs<ST, CT, PAR>(pdf, N, c, D, f);
    moments_of<ST, CT>(f, (CT)eps[c], (CT)fpf[c], (CT)fpf[N + c], (CT)fpf[2 * N + c], fbx, fby, fbz, o);
    rho_o[c] = (FT)o[0];
    ire[c] = (FT)o[4];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        j_o[a * N + c] = (FT)o[1 + a];
        uD[a * N + c] = (FT)o[5 + a];
    }
}

// the cells c and c + 1, as in K1: every plane that keeps the pair aligned moves
// as a two-element vector: K2a and K2b together 1.07 -> 0.60 ms (256^3, FP16
// storage), 0.43 -> 0.30 ms (192^3, FP32)
template <typename ST, typename FT, typename CT, int PAR>
__device__ __forceinline__ void moments_pair(const ST *__restrict__ pdf, const FT *__restrict__ eps,
                                             const FT *__restrict__ fpf, const Geom &g, long long c, CT fbx, CT fby,
                                             CT fbz, FT *__restrict__ rho_o, FT *__restrict__ j_o,
                                             FT *__restrict__ uD, FT *__restrict__ ire) {
    const unsigned N = (unsigned)g.ncell, cu = (unsigned)c;
    NbDelta D, D1;
    if (PAR) {
        int ix, iy, iz;
        cell_coords(g, c, ix, iy, iz);
        D = neighbour_deltas(g, ix, iy, iz);
        D1 = neighbour_deltas(g, ix + 1, iy, iz);
        if (!no_wall_neighbour(D) || !no_wall_neighbour(D1)) {
            moments_cell<ST, FT, CT, PAR>(pdf, eps, fpf, g, c, fbx, fby, fbz, rho_o, j_o, uD, ire);
            moments_cell<ST, FT, CT, PAR>(pdf, eps, fpf, g, c + 1, fbx, fby, fbz, rho_o, j_o, uD, ire);
            return;
        }
    }
    CT f[Q], f1[Q], e0, e1, a[3], b[3], o[8], o1[8];
    load_pair<ST, CT, PAR>(pdf, N, cu, D, D1, f, f1);
    Vec2<FT>::load(eps + cu, e0, e1);
#pragma unroll
    for (int k = 0; k < 3; ++k) Vec2<FT>::load(fpf + (k * N + cu), a[k], b[k]);
    moments_of<ST, CT>(f, e0, a[0], a[1], a[2], fbx, fby, fbz, o);
    moments_of<ST, CT>(f1, e1, b[0], b[1], b[2], fbx, fby, fbz, o1);
    Vec2<FT>::store(rho_o + cu, o[0], o1[0]);
    Vec2<FT>::store(ire + cu, o[4], o1[4]);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        Vec2<FT>::store(j_o + (k * N + cu), o[1 + k], o1[1 + k]);
        Vec2<FT>::store(uD + (k * N + cu), o[5 + k], o1[5 + k]);
    }
}

#ifndef DPS_MOM_MINB
#define DPS_MOM_MINB 3  // FP64: 128-thread blocks per SM the register budget is sized for
#endif
template <typename ST, typename FT, typename CT, int PAR>
__global__ void __launch_bounds__(128, sizeof(CT) == 8 ? DPS_MOM_MINB : 4) k_moments(const BoxDev *__restrict__ boxes,
                                                    const Tile *__restrict__ tiles, int ntiles) {
    DPS_FOR_TILES(tiles, ntiles, t) {
        const Tile tl = tiles[t];
        const BoxDev &B = boxes[tl.box];
        const Geom g = B.g;
        const ST *pdf = (const ST *)B.pdf;
        const FT *eps = (const FT *)B.eps, *fpf = (const FT *)B.fpf;
        FT *rho = (FT *)B.rho, *j = (FT *)B.j, *uD = (FT *)B.uD, *ire = (FT *)B.ire;
        const CT fbx = pick<CT>(B.ph.fb[0], B.ph.fb_f[0]), fby = pick<CT>(B.ph.fb[1], B.ph.fb_f[1]),
                 fbz = pick<CT>(B.ph.fb[2], B.ph.fb_f[2]);
        if constexpr (sizeof(ST) < 8)
            if (!(g.ncell & 1) && !((tl.begin | tl.end) & 1) && (!PAR || !(g.n[0] & 1))) {
                for (long long c = tl.begin + 2 * threadIdx.x; c < tl.end; c += 2 * blockDim.x)
                    moments_pair<ST, FT, CT, PAR>(pdf, eps, fpf, g, c, fbx, fby, fbz, rho, j, uD, ire);
                continue;
            }
        for (long long c = tl.begin + threadIdx.x; c < tl.end; c += blockDim.x)
            moments_cell<ST, FT, CT, PAR>(pdf, eps, fpf, g, c, fbx, fby, fbz, rho, j, uD, ire);
    }
}

// K2b: grad P with P = eps_f p = c_s^2 rho, and Du_f/Dt = (u_D - u_prev) +
// (u_D . grad) u_D, with the lattice gradient of Sec. 3.2.3.  Neighbours
// beyond a wall are mirrored into the box (coordinate clamped).
#ifndef DPS_FIELDS32_MINB
#define DPS_FIELDS32_MINB 8  // 256-thread blocks per SM the register budget is sized for
#endif
constexpr int FB = 8, FH = FB + 2, FH3 = FH * FH * FH;

// coordinate of the cell at i on axis a, wrapped or mirrored
__device__ __forceinline__ int near_cell(const Geom &g, int a, int i) {
    if (i < 0) return g.per[a] ? g.n[a] - 1 : 0;
    if (i >= g.n[a]) return g.per[a] ? 0 : g.n[a] - 1;
    return i;
}

// The FP32 forms over bricks of 8^3 cells: rho and u_D of the brick and its
// halo are staged in shared memory as one float4 a cell, so a neighbour is one
// 16-byte load off a constant offset and not four words of global memory with
// a 64-bit address: K2a and K2b together 1.53 -> 1.07 ms (256^3, FP16 storage),
// 0.66 -> 0.44 ms (192^3, FP32).  Each sum keeps the order of q.
__global__ void __launch_bounds__(256, DPS_FIELDS32_MINB) k_fields32(const BoxDev *__restrict__ boxes,
                                                                      const Tile *__restrict__ tiles, int ntiles) {
    __shared__ float4 S[FH3];
    DPS_FOR_TILES(tiles, ntiles, t) {
        const Tile tl = tiles[t];
        const BoxDev &B = boxes[tl.box];
        const Geom g = B.g;
        const long long N = g.ncell;
        int ox, oy, oz, ex, ey, ez;
        brick_of(tl, ox, oy, oz, ex, ey, ez);
        const float *rho = (const float *)B.rho, *uD = (const float *)B.uD;
        float *uprev = (float *)B.uprev, *gradP = (float *)B.gradP, *DuDt = (float *)B.DuDt;
        const int have_prev = B.have_uprev;
        __syncthreads();  // the previous brick is done with S
        for (int h = threadIdx.x; h < FH3; h += 256) {
            const int hx = h % FH, hy = (h / FH) % FH, hz = h / (FH * FH);
            if (hx > ex + 1 || hy > ey + 1 || hz > ez + 1) continue;
            const long long n = cell_index(g, near_cell(g, 0, ox + hx - 1), near_cell(g, 1, oy + hy - 1),
                                           near_cell(g, 2, oz + hz - 1));
            S[h] = make_float4(rho[n], uD[n], uD[N + n], uD[2 * N + n]);
        }
        __syncthreads();
        const int nb = ex * ey * ez;
        for (int k = threadIdx.x; k < nb; k += 256) {
            const int lx = k % ex, ly = (k / ex) % ey, lz = k / (ex * ey);
            const long long c = cell_index(g, ox + lx, oy + ly, oz + lz);
            const int p = ((lz + 1) * FH + ly + 1) * FH + lx + 1;
            const float4 s = S[p];
            const float u[3] = {s.y, s.z, s.w};
            float up[3];
#pragma unroll
            for (int b = 0; b < 3; ++b) up[b] = have_prev ? uprev[b * N + c] : u[b];
            float gp[3] = {0, 0, 0};
            float gu[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};  // gu[a][b] = sum w c_a u_b
#pragma unroll
            for (int q = 1; q < Q; ++q) {
                const float4 v = S[p + (CZ(q) * FH + CY(q)) * FH + CX(q)];
                const float w = (float)WQ(q);
                const int cc[3] = {CX(q), CY(q), CZ(q)};
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    if (cc[a] == 0) continue;
                    const float wc = w * (float)cc[a];
                    gp[a] += wc * v.x;
                    gu[a][0] += wc * v.y;
                    gu[a][1] += wc * v.z;
                    gu[a][2] += wc * v.w;
                }
            }
            // c_s^-2 sum w c phi; for P = c_s^2 rho the c_s^2 cancels
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                gradP[b * N + c] = gp[b];
                const float conv = 3.0f * (u[0] * gu[0][b] + u[1] * gu[1][b] + u[2] * gu[2][b]);
                DuDt[b * N + c] = (u[b] - up[b]) + conv;
                uprev[b * N + c] = u[b];
            }
        }
    }
}

// K2b of the FP64 form over bricks of 8^3 cells: rho and u_D of the brick and its
// halo are staged in shared memory as integers of 58 bits relative to the
// largest of the block (rho apart from u_D), so that the 18-neighbour sums are
// exact integer additions and the convective products 64-bit ones; 12 FP64
// instructions a cell are left of 135, which bound this kernel.  A block with a
// non-finite value takes FP64 throughout.  K2a and K2b together at 256^3: 6.34
// -> 2.12 ms; at 64^3: 115 -> 46 us.

__device__ __forceinline__ void fields_cell64(const double *__restrict__ rho, const double *__restrict__ uD,
                                              const Geom &g, int ix, int iy, int iz, double gp[3], double cv[3]) {
    const long long N = g.ncell, c = cell_index(g, ix, iy, iz);
    const int ii[3] = {ix, iy, iz};
    double gu[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
    gp[0] = gp[1] = gp[2] = 0.0;
#pragma unroll 1
    for (int q = 1; q < Q; ++q) {
        const int cc[3] = {CX(q), CY(q), CZ(q)};
        int t[3];
        for (int a = 0; a < 3; ++a) {
            t[a] = ii[a] + cc[a];
            if (t[a] < 0) t[a] = g.per[a] ? g.n[a] - 1 : 0;
            if (t[a] >= g.n[a]) t[a] = g.per[a] ? 0 : g.n[a] - 1;
        }
        const long long n = cell_index(g, t[0], t[1], t[2]);
        const double r = rho[n], u0 = uD[n], u1 = uD[N + n], u2 = uD[2 * N + n];
        for (int a = 0; a < 3; ++a) {
            const double wc = WQ(q) * cc[a];
            gp[a] += wc * r;
            gu[a][0] += wc * u0;
            gu[a][1] += wc * u1;
            gu[a][2] += wc * u2;
        }
    }
    const double u[3] = {uD[c], uD[N + c], uD[2 * N + c]};
    for (int b = 0; b < 3; ++b) cv[b] = 3.0 * (u[0] * gu[0][b] + u[1] * gu[1][b] + u[2] * gu[2][b]);
}

// 36 sum_q w_q c_q phi(x + c_q) at entry p of the staged field
__device__ __forceinline__ void stencil36(const i64 *__restrict__ s, int p, i64 G[3]) {
    constexpr int Y = FH, Z = FH * FH;
    const i64 xpyp = s[p + 1 + Y], xpym = s[p + 1 - Y], xmyp = s[p - 1 + Y], xmym = s[p - 1 - Y];
    const i64 xpzp = s[p + 1 + Z], xpzm = s[p + 1 - Z], xmzp = s[p - 1 + Z], xmzm = s[p - 1 - Z];
    const i64 ypzp = s[p + Y + Z], ypzm = s[p + Y - Z], ymzp = s[p - Y + Z], ymzm = s[p - Y - Z];
    G[0] = 2 * (s[p + 1] - s[p - 1]) + (xpyp - xmym) + (xpym - xmyp) + (xpzp - xmzm) + (xpzm - xmzp);
    G[1] = 2 * (s[p + Y] - s[p - Y]) + (xpyp - xmym) - (xpym - xmyp) + (ypzp - ymzm) + (ypzm - ymzp);
    G[2] = 2 * (s[p + Z] - s[p - Z]) + (xpzp - xmzm) - (xpzm - xmzp) + (ypzp - ymzm) - (ypzm - ymzp);
}

__global__ void __launch_bounds__(256) k_fields64(const BoxDev *__restrict__ boxes, const Tile *__restrict__ tiles,
                                                  int ntiles) {
    __shared__ i64 S[4][FH3];
    __shared__ u32 top[2];
    DPS_FOR_TILES(tiles, ntiles, t) {
        const Tile tl = tiles[t];
        const BoxDev &B = boxes[tl.box];
        const Geom g = B.g;
        const long long N = g.ncell;
        int ox, oy, oz, ex, ey, ez;
        brick_of(tl, ox, oy, oz, ex, ey, ez);
        const double *rho = (const double *)B.rho, *uD = (const double *)B.uD;
        if (threadIdx.x < 2) top[threadIdx.x] = 0;
        __syncthreads();  // (also: the previous brick is done with S)
        // stage the raw bits and the largest exponents (neighbours beyond a
        // wall are mirrored into the box: coordinate clamped)
        u32 mr = 0, mu = 0;
        for (int h = threadIdx.x; h < FH3; h += 256) {
            const int hx = h % FH, hy = (h / FH) % FH, hz = h / (FH * FH);
            u64 v[4] = {0, 0, 0, 0};
            if (hx <= ex + 1 && hy <= ey + 1 && hz <= ez + 1) {
                const long long n = cell_index(g, near_cell(g, 0, ox + hx - 1), near_cell(g, 1, oy + hy - 1),
                                               near_cell(g, 2, oz + hz - 1));
                v[0] = fx_bits(rho[n]);
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    v[1 + k] = fx_bits(uD[k * N + n]);
                    mu = max(mu, fx_abs_hi(v[1 + k]));
                }
                mr = max(mr, fx_abs_hi(v[0]));
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) S[k][h] = (i64)v[k];
        }
        mr = __reduce_max_sync(0xffffffffu, mr);
        mu = __reduce_max_sync(0xffffffffu, mu);
        if ((threadIdx.x & 31) == 0) {
            atomicMax(&top[0], mr);
            atomicMax(&top[1], mu);
        }
        __syncthreads();
        // |v| < 2^(e + 1): units of 2^(e - 57) leave four bits for the sums
        const int er = (int)(top[0] >> 20) - 1023, eu = max((int)(top[1] >> 20) - 1023, -400);
        const bool fixed = er < 1024 && er > -400 && eu < 400;
        const int fr = 57 - er, fu = 57 - eu;
        if (fixed) {
            for (int h = threadIdx.x; h < FH3; h += 256) {
                S[0][h] = fx_from(fx_double((u64)S[0][h]), fr);
#pragma unroll
                for (int k = 1; k < 4; ++k) S[k][h] = fx_from(fx_double((u64)S[k][h]), fu);
            }
        }
        __syncthreads();
        double *uprev = (double *)B.uprev, *gradP = (double *)B.gradP, *DuDt = (double *)B.DuDt;
        const int have_prev = B.have_uprev;
        const int nb = ex * ey * ez;
        for (int k = threadIdx.x; k < nb; k += 256) {
            const int lx = k % ex, ly = (k / ex) % ey, lz = k / (ex * ey);
            const long long c = cell_index(g, ox + lx, oy + ly, oz + lz);
            double gp[3], cv[3], u[3];
#pragma unroll
            for (int b = 0; b < 3; ++b) u[b] = uD[b * N + c];
            if (fixed) {
                const int p = ((lz + 1) * FH + ly + 1) * FH + lx + 1;
                i64 G[3];
                stencil36(S[0], p, G);
#pragma unroll
                for (int b = 0; b < 3; ++b) gp[b] = fx_signed_to_double(G[b], fr) * (1.0 / 36.0);
                const i64 v[3] = {S[1][p] * 16, S[2][p] * 16, S[3][p] * 16};
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                    stencil36(S[1 + b], p, G);
                    // (u . grad) u_b = 3/36 sum_a u_a G_a: three products of the high halves
                    const i64 C = fx_mulhi_s(v[0], G[0]) + fx_mulhi_s(v[1], G[1]) + fx_mulhi_s(v[2], G[2]) + 1;
                    cv[b] = fx_signed_to_double(C, 2 * fu + 4 - 64) * (1.0 / 12.0);
                }
            } else {
                fields_cell64(rho, uD, g, ox + lx, oy + ly, oz + lz, gp, cv);
            }
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                gradP[b * N + c] = gp[b];
                const double up = have_prev ? uprev[b * N + c] : u[b];
                DuDt[b * N + c] = (u[b] - up) + cv[b];
                uprev[b * N + c] = u[b];
            }
        }
    }
}

// Lift support (Table 1, Sec. 3.2.3): curl of the fluid velocity at the
// subcycle start, u_f = (j + eps_f f_b / 2)/(rho eps_f) with the current eps_f,
// by the lattice rule curl psi = c_s^-2 sum_q w_q c_q x psi(x + c_q) (walls:
// neighbour coordinate clamped, as for the gradient).  u_f of a neighbour is
// evaluated on the fly from rho, j and eps_f; boxes without lift are skipped.
template <typename FT, typename CT>
__global__ void __launch_bounds__(256) k_curl(const BoxDev *__restrict__ boxes, const Tile *__restrict__ tiles,
                                              int ntiles) {
    DPS_FOR_TILES(tiles, ntiles, t) {
        const Tile tl = tiles[t];
        const BoxDev &B = boxes[tl.box];
        if (!B.ph.lift || B.np == 0) continue;
        const Geom g = B.g;
        const long long N = g.ncell;
        const FT *rho = (const FT *)B.rho, *j = (const FT *)B.j, *eps = (const FT *)B.eps;
        FT *curl = (FT *)B.curl;
        const CT hb[3] = {CT(0.5) * (CT)B.ph.fb[0], CT(0.5) * (CT)B.ph.fb[1], CT(0.5) * (CT)B.ph.fb[2]};
        for (long long c = tl.begin + threadIdx.x; c < tl.end; c += blockDim.x) {
            int ix, iy, iz;
            cell_coords(g, c, ix, iy, iz);
            long long stride[3] = {1, g.n[0], (long long)g.n[0] * g.n[1]};
            const int ii[3] = {ix, iy, iz};
            long long dd[3][3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                int L = g.n[a];
                dd[a][1] = 0;
                dd[a][0] = ii[a] > 0 ? -stride[a] : (g.per[a] ? (long long)(L - 1) * stride[a] : 0);
                dd[a][2] = ii[a] < L - 1 ? stride[a] : (g.per[a] ? -(long long)(L - 1) * stride[a] : 0);
            }
            CT r[3] = {0, 0, 0};
#pragma unroll
            for (int q = 1; q < Q; ++q) {
                const long long n = c + dd[0][CX(q) + 1] + dd[1][CY(q) + 1] + dd[2][CZ(q) + 1];
                const CT e = (CT)eps[n];
                const CT sc = CT(1) / ((CT)rho[n] * e);
                const CT v0 = ((CT)j[n] + e * hb[0]) * sc;
                const CT v1 = ((CT)j[N + n] + e * hb[1]) * sc;
                const CT v2 = ((CT)j[2 * N + n] + e * hb[2]) * sc;
                const CT w = CT(3) * (CT)WQ(q);
                if (CY(q) != 0 || CZ(q) != 0) r[0] += w * (CT(CY(q)) * v2 - CT(CZ(q)) * v1);
                if (CZ(q) != 0 || CX(q) != 0) r[1] += w * (CT(CZ(q)) * v0 - CT(CX(q)) * v2);
                if (CX(q) != 0 || CY(q) != 0) r[2] += w * (CT(CX(q)) * v1 - CT(CY(q)) * v0);
            }
#pragma unroll
            for (int a = 0; a < 3; ++a) curl[a * N + c] = (FT)r[a];
        }
    }
}

// The FP64 form over bricks of 8^3 cells, as k_fields64: u_f is evaluated once per
// staged cell (18 divisions a cell otherwise bound the kernel), brought to
// integers of 58 bits relative to the block's largest component, and the curl is
// exact integer sums.  u_f itself goes to the f_pf,am planes (free until the
// reaction is gathered) for the interpolation of the lift.  75 x 61 x 90, two
// subcycles: curl and added-mass passes 0.76 -> 0.24 ms a step.
__global__ void __launch_bounds__(256) k_curl64(const BoxDev *__restrict__ boxes, const Tile *__restrict__ tiles,
                                                int ntiles) {
    __shared__ i64 S[3][FH3];
    __shared__ u32 top;
    DPS_FOR_TILES(tiles, ntiles, t) {
        const Tile tl = tiles[t];
        const BoxDev &B = boxes[tl.box];
        if (!B.ph.lift || B.np == 0) continue;
        const Geom g = B.g;
        const long long N = g.ncell;
        int ox, oy, oz, ex, ey, ez;
        brick_of(tl, ox, oy, oz, ex, ey, ez);
        const double *rho = (const double *)B.rho, *j = (const double *)B.j, *eps = (const double *)B.eps;
        const double hb[3] = {0.5 * B.ph.fb[0], 0.5 * B.ph.fb[1], 0.5 * B.ph.fb[2]};
        double *uf = (double *)B.fam, *curl = (double *)B.curl;
        if (threadIdx.x == 0) top = 0;
        __syncthreads();  // (also: the previous brick is done with S)
        u32 mu = 0;
        for (int h = threadIdx.x; h < FH3; h += 256) {
            const int hx = h % FH, hy = (h / FH) % FH, hz = h / (FH * FH);
            u64 v[3] = {0, 0, 0};
            if (hx <= ex + 1 && hy <= ey + 1 && hz <= ez + 1) {
                int p[3] = {ox + hx - 1, oy + hy - 1, oz + hz - 1};
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    if (p[a] < 0) p[a] = g.per[a] ? g.n[a] - 1 : 0;
                    else if (p[a] >= g.n[a]) p[a] = g.per[a] ? 0 : g.n[a] - 1;
                }
                const long long n = cell_index(g, p[0], p[1], p[2]);
                const double e = eps[n], r = rho[n];
                double q;
                if (r > 0.5 && r < 2.0 && e > 0.125 && e <= 1.0) {
                    int lz;
                    const u64 R = fx_recip(fx_q62(fx_bits(r)), fx_from_pos(e, 62), lz);
                    q = fx_to_double(R, 64 - lz);
                } else {
                    q = 1.0 / (r * e);
                }
                const bool own = hx >= 1 && hx <= ex && hy >= 1 && hy <= ey && hz >= 1 && hz <= ez;
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const double u = (j[k * N + n] + e * hb[k]) * q;
                    if (own) uf[k * N + n] = u;
                    v[k] = fx_bits(u);
                    mu = max(mu, fx_abs_hi(v[k]));
                }
            }
#pragma unroll
            for (int k = 0; k < 3; ++k) S[k][h] = (i64)v[k];
        }
        mu = __reduce_max_sync(0xffffffffu, mu);
        if ((threadIdx.x & 31) == 0) atomicMax(&top, mu);
        __syncthreads();
        const int eu = max((int)(top >> 20) - 1023, -400), fu = 57 - eu;
        const bool fixed = eu < 400;  // else: a value is not finite (or the run is past all bounds)
        if (fixed)
            for (int h = threadIdx.x; h < FH3; h += 256)
#pragma unroll
                for (int k = 0; k < 3; ++k) S[k][h] = fx_from(fx_double((u64)S[k][h]), fu);
        __syncthreads();
        const int nb = ex * ey * ez;
        for (int k = threadIdx.x; k < nb; k += 256) {
            const int lx = k % ex, ly = (k / ex) % ey, lz = k / (ex * ey);
            const long long c = cell_index(g, ox + lx, oy + ly, oz + lz);
            const int p = ((lz + 1) * FH + ly + 1) * FH + lx + 1;
            double r[3];
            if (fixed) {
                i64 X[3], Y[3], Z[3];
                stencil36(S[0], p, X);
                stencil36(S[1], p, Y);
                stencil36(S[2], p, Z);
                r[0] = fx_signed_to_double(Z[1] - Y[2], fu) * (1.0 / 12.0);
                r[1] = fx_signed_to_double(X[2] - Z[0], fu) * (1.0 / 12.0);
                r[2] = fx_signed_to_double(Y[0] - X[1], fu) * (1.0 / 12.0);
            } else {  // S holds the bits of u_f
                r[0] = r[1] = r[2] = 0.0;
#pragma unroll 1
                for (int q = 1; q < Q; ++q) {
                    const int n = p + (CZ(q) * FH + CY(q)) * FH + CX(q);
                    const double u0 = fx_double((u64)S[0][n]), u1 = fx_double((u64)S[1][n]), u2 = fx_double((u64)S[2][n]);
                    const double w = 3.0 * WQ(q);
                    r[0] += w * (CY(q) * u2 - CZ(q) * u1);
                    r[1] += w * (CZ(q) * u0 - CX(q) * u2);
                    r[2] += w * (CX(q) * u1 - CY(q) * u0);
                }
            }
#pragma unroll
            for (int a = 0; a < 3; ++a) curl[a * N + c] = r[a];
        }
    }
}

// ---- canonical PDF export / import (FP64 host view) -------------------------
template <typename ST, int PAR>
__global__ void k_pdf_export(const ST *__restrict__ pdf, Geom g, double *__restrict__ out) {
    const long long N = g.ncell;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N;
         c += (long long)gridDim.x * blockDim.x) {
        int ix, iy, iz;
        cell_coords(g, c, ix, iy, iz);
        NbDelta D = neighbour_deltas(g, ix, iy, iz);
        if constexpr (sizeof(ST) == 8) {
            double f[Q];
            load_pdfs<ST, double, PAR>(pdf, N, c, D, f);
#pragma unroll
            for (int q = 0; q < Q; ++q) out[(long long)q * N + c] = f[q];
        } else {
            float f[Q];
            load_pdfs<ST, float, PAR>(pdf, N, c, D, f);
#pragma unroll
            for (int q = 0; q < Q; ++q) out[(long long)q * N + c] = (double)f[q] + WQ(q);
        }
    }
}

// import always writes the even (canonical) layout
template <typename ST>
__global__ void k_pdf_import(ST *__restrict__ pdf, long long N, const double *__restrict__ in) {
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < N;
         c += (long long)gridDim.x * blockDim.x) {
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            if constexpr (sizeof(ST) == 8)
                Store<ST>::store(pdf + (long long)q * N + c, in[(long long)q * N + c]);
            else  // shifted storage: the deviation is taken in FP64, then rounded
                Store<ST>::store(pdf + (long long)q * N + c, (float)(in[(long long)q * N + c] - WQ(q)));
        }
    }
}

// ---- host launchers ----------------------------------------------------------
static int grid_for(long long n, int block) {
    long long g = (n + block - 1) / block;
    long long cap = 152LL * 16;  // grid-stride beyond this
    if (g > cap) g = cap;
    return (int)(g < 1 ? 1 : g);
}

// variant: register budget of K1 (blocks of 128 threads per SM the compiler
// must fit) and cells per thread (variants 3, 4, 5: two; 6, 7: two adjacent
// cells moved as two-element vectors); chosen by the batch
// autotuner.  visc: some box of the batch
// relaxes with a per-cell tau_e (one register budget for that variant).
template <typename ST, typename FT, typename CT>
void launch_collide_stream(const BoxDev *boxes, const Tile *tiles, int ntiles, int parity, int variant, bool visc, int grid, int block, cudaStream_t s) {
    block = 128;
    if (sizeof(CT) == 8) variant = 0;  // FP64: one register-heavy variant
#define DPS_K1V(MB, V, CPT)                                                                           \
    do {                                                                                                  \
        if (parity)                                                                                       \
            k_collide_stream<ST, FT, CT, 1, MB, V, CPT><<<grid, block, 0, s>>>(boxes, tiles, ntiles);  \
        else                                                                                              \
            k_collide_stream<ST, FT, CT, 0, MB, V, CPT><<<grid, block, 0, s>>>(boxes, tiles, ntiles);  \
    } while (0)
#define DPS_K1(MB, CPT) DPS_K1V(MB, false, CPT)
    if constexpr (sizeof(CT) == 8) {
        if (visc) DPS_K1V(DPS_K1V_MINB, true, 1);
        else DPS_K1(DPS_K1_MINB, 1);
    } else if (visc)
        DPS_K1V(3, true, 1);
    else if (variant == 1)
        DPS_K1(3, 1);
    else if (variant == 2)
        DPS_K1(5, 1);
    else if (variant == 3)
        DPS_K1(3, 2);
    else if (variant == 4)
        DPS_K1(4, 2);
    else if (variant == 5)
        DPS_K1(2, 2);
    else if (variant == 6)
        DPS_K1(4, 3);
    else if (variant == 7)
        DPS_K1(3, 3);
    else
        DPS_K1(4, 1);
#undef DPS_K1
#undef DPS_K1V
}

template <typename ST, typename FT, typename CT>
void launch_moments(const BoxDev *boxes, const Tile *tiles, int ntiles, int parity, int grid, int block,
                    cudaStream_t s) {
    if (block > 128) block = 128;
    if (parity)
        k_moments<ST, FT, CT, 1><<<grid, block, 0, s>>>(boxes, tiles, ntiles);
    else
        k_moments<ST, FT, CT, 0><<<grid, block, 0, s>>>(boxes, tiles, ntiles);
}

void launch_fields64(const BoxDev *boxes, const Tile *bricks, int nbricks, cudaStream_t s) {
    k_fields64<<<nbricks, 256, 0, s>>>(boxes, bricks, nbricks);
}
void launch_fields32(const BoxDev *boxes, const Tile *bricks, int nbricks, cudaStream_t s) {
    k_fields32<<<nbricks, 256, 0, s>>>(boxes, bricks, nbricks);
}

void launch_curl64(const BoxDev *boxes, const Tile *bricks, int nbricks, cudaStream_t s) {
    k_curl64<<<nbricks, 256, 0, s>>>(boxes, bricks, nbricks);
}
void launch_curl32(const BoxDev *boxes, const Tile *tiles, int ntiles, int grid, int block, cudaStream_t s) {
    k_curl<float, float><<<grid, block, 0, s>>>(boxes, tiles, ntiles);
}

template <typename ST>
void launch_pdf_export(const void *pdf, const Geom &g, int parity, double *out, cudaStream_t s) {
    const int B = 128;
    if (parity == 0)
        k_pdf_export<ST, 0><<<grid_for(g.ncell, B), B, 0, s>>>((const ST *)pdf, g, out);
    else
        k_pdf_export<ST, 1><<<grid_for(g.ncell, B), B, 0, s>>>((const ST *)pdf, g, out);
}

template <typename ST>
void launch_pdf_import(void *pdf, long long N, const double *in, cudaStream_t s) {
    const int B = 128;
    k_pdf_import<ST><<<grid_for(N, B), B, 0, s>>>((ST *)pdf, N, in);
}

// explicit instantiations for the three precision forms
#define DPS_LBM_INST(ST, FT, CT)                                                                             \
    template void launch_collide_stream<ST, FT, CT>(const BoxDev *, const Tile *, int, int, int, bool, int, int, cudaStream_t); \
    template void launch_moments<ST, FT, CT>(const BoxDev *, const Tile *, int, int, int, int, cudaStream_t);
DPS_LBM_INST(double, double, double)
DPS_LBM_INST(float, float, float)
DPS_LBM_INST(__half, float, float)
template void launch_pdf_export<double>(const void *, const Geom &, int, double *, cudaStream_t);
template void launch_pdf_export<float>(const void *, const Geom &, int, double *, cudaStream_t);
template void launch_pdf_export<__half>(const void *, const Geom &, int, double *, cudaStream_t);
template void launch_pdf_import<double>(void *, long long, const double *, cudaStream_t);
template void launch_pdf_import<float>(void *, long long, const double *, cudaStream_t);
template void launch_pdf_import<__half>(void *, long long, const double *, cudaStream_t);

}  // namespace dps
