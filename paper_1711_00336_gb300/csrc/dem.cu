// dem.cu -- S6: the DEM substeps of Algorithm 1.
//
// Per particle (cell-sorted order): contact (Sec. 3.1.1, linear spring-dashpot
// with Coulomb-capped viscous friction), lubrication (Sec. 3.1.3, Ball &
// Melrose) against neighbours and walls, then the explicit update of Eq.
// particle_motion with the frozen F_fp + F_g.
//
// Neighbour list: after every sort a Verlet list is built per particle from
// the linked cells of the +-R cells around it, keeping every partner within
// the interaction range plus the skin; the n_DEM substeps then loop over the
// list only.  FP64 form: each pair of the list is evaluated once per substep
// (k_dem_pairs64; lubrication pairs in 64-bit integer arithmetic of more than
// FP64's precision, fx.cuh) and a gather kernel adds it to both partners in an
// order fixed by the list (k_dem_gather64).  Mixed forms: a substep gives each
// particle a group of LANES consecutive lanes of a warp: lane l takes the list
// entries l, l + LANES, ... and the group's force and torque sums are combined
// by warp shuffles (a fixed xor tree, so the result does not depend on the
// launch shape); one thread per particle then adds the walls and integrates.
// A particle that moves more than skin/2 before the next sort raises
// DPS_ERR_UNSTABLE.  Candidate distances are screened in FP32 (a float
// copy of the positions, refreshed every substep, with a margin far above its
// rounding) and every pair that passes is evaluated: in FP64 for the FP64
// form, and in FP32 for the low-precision forms, where a pair close to
// contact (gap below 1e-3 dx or overlap) takes its separation from the FP64
// positions.  Positions, velocities and the integration are FP64 in every
// form.  State is read from one buffer and
// written to the other (ping-pong), so every pair sees the substep start.
#include "box.cuh"

namespace dps {

static constexpr double PI_D = 3.14159265358979323846;
static constexpr float SCREEN_MARGIN = 1e-3f;  // >> FP32 rounding of positions < 2^16 cells
static constexpr double H_NEAR = 1e-3;         // gaps below this: separation from the FP64 positions (mixed forms)

// minimum image for |dx| < L (positions live in [0, L))
__device__ __forceinline__ double min_image(double dx, int L, int per) {
    if (!per) return dx;
    const double h = 0.5 * L;
    return dx > h ? dx - L : (dx < -h ? dx + L : dx);
}
__device__ __forceinline__ float min_image_f(float dx, float L, int per) {
    if (!per) return dx;
    const float h = 0.5f * L;
    return dx > h ? dx - L : (dx < -h ? dx + L : dx);
}

template <typename T>
__device__ __forceinline__ void cross3(const T a[3], const T b[3], T o[3]) {
    o[0] = a[1] * b[2] - a[2] * b[1];
    o[1] = a[2] * b[0] - a[0] * b[2];
    o[2] = a[0] * b[1] - a[1] * b[0];
}

// closure constants of the pair forces in arithmetic T, converted once per
// tile (no FP64 conversions inside the FP32 pair loop)
template <typename T>
struct PairPar {
    T kfac, xfac, mu_c, h_c, h_min, mu, capfac;
    int contact, lubrication, lub_limiter;
};
template <typename T>
__device__ __forceinline__ PairPar<T> pair_par(const Phys &ph) {
    PairPar<T> q;
    q.kfac = (T)ph.kfac;
    q.xfac = (T)ph.xfac;
    q.mu_c = (T)ph.mu_c;
    q.h_c = (T)ph.h_c;
    q.h_min = (T)ph.h_min;
    q.mu = (T)ph.mu;
    q.capfac = (T)ph.capfac;
    q.contact = ph.contact;
    q.lubrication = ph.lubrication;
    q.lub_limiter = ph.lub_limiter;
    return q;
}

// spring-dashpot contact with Coulomb friction (Sec. 3.1.1) for overlap
// delta > 0, in arithmetic T, accumulated in T; the torque is
// (d_i/2) n x F_t (r x F at the contact point r = d_i/2 n).
// lev: the lever of the torque, d_i/2 (or 1, which leaves n x F_t in Tq for
// the pair kernel of the FP64 form: both partners take it times their d/2)
template <typename T>
__device__ __forceinline__ void contact_force(const PairPar<T> &ph, const T n[3], T delta, const T ui[3],
                                              const T wi[3], T di, const T uj[3], const T wjh[3], T m_ij, T lev,
                                              T F[3], T Tq[3]) {
    // k_n and xi_n of Eqs. damping_to_stiffness / collision_time, solved
    // for the given e_n and T_c: both proportional to m_ij
    const T k_n = m_ij * ph.kfac;
    const T xi = m_ij * ph.xfac;
    T ws[3], wx[3], ur[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) ws[a] = T(0.5) * di * wi[a] + wjh[a];
    cross3(ws, n, wx);
#pragma unroll
    for (int a = 0; a < 3; ++a) ur[a] = ui[a] - uj[a] + wx[a];
    const T urn = ur[0] * n[0] + ur[1] * n[1] + ur[2] * n[2];
    T ut[3], Fn[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        ut[a] = ur[a] - urn * n[a];
        Fn[a] = -k_n * delta * n[a] - xi * (urn * n[a]);
    }
    const T Fn_abs = m_sqrt(Fn[0] * Fn[0] + Fn[1] * Fn[1] + Fn[2] * Fn[2]);
    const T ut_abs = m_sqrt(ut[0] * ut[0] + ut[1] * ut[1] + ut[2] * ut[2]);
    T Ft[3] = {0, 0, 0};
    if (ut_abs > T(0)) {
        const T mag = m_min(ph.mu_c * Fn_abs, xi * ut_abs) / ut_abs;
#pragma unroll
        for (int a = 0; a < 3; ++a) Ft[a] = -mag * ut[a];
    }
    T nF[3];
    cross3(n, Ft, nF);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        F[a] += Fn[a] + Ft[a];
        Tq[a] += lev * nF[a];
    }
}

// the FP64 form of it: |F_n| = |k_n delta + xi u_n| since n is a unit vector,
// and the friction is xi u_t unless mu_c |F_n| caps it, so the square root and
// the divisions of the general form shrink to one reciprocal square root on
// the sliding branch (an FP64 square root or division costs ~8.5 multiply-adds)
__device__ __forceinline__ void contact_force(const PairPar<double> &ph, const double n[3], double delta,
                                              const double ui[3], const double wi[3], double di, const double uj[3],
                                              const double wjh[3], double m_ij, double lev, double F[3], double Tq[3]) {
    double ws[3], wx[3], ur[3], ut[3], Ft[3], nF[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) ws[a] = 0.5 * di * wi[a] + wjh[a];
    cross3(ws, n, wx);
#pragma unroll
    for (int a = 0; a < 3; ++a) ur[a] = ui[a] - uj[a] + wx[a];
    const double urn = ur[0] * n[0] + ur[1] * n[1] + ur[2] * n[2];
    const double xi = m_ij * ph.xfac, fn = m_ij * ph.kfac * delta + xi * urn;
#pragma unroll
    for (int a = 0; a < 3; ++a) ut[a] = ur[a] - urn * n[a];
    const double ut2 = ut[0] * ut[0] + ut[1] * ut[1] + ut[2] * ut[2];
    const double lim = ph.mu_c * fabs(fn);
    double mag = xi;
    if (!(xi * xi * ut2 <= lim * lim)) mag = lim * rsqrt(ut2);
#pragma unroll
    for (int a = 0; a < 3; ++a) Ft[a] = -mag * ut[a];
    cross3(n, Ft, nF);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        F[a] += Ft[a] - fn * n[a];
        Tq[a] += lev * nF[a];
    }
}

// lubrication correction (Sec. 3.1.3) at the floored gap hh, given <d>,
// r = <d>/hh, ir = 1/r and the limiter cap m_ij capfac
template <typename T>
__device__ __forceinline__ void lub_force(const PairPar<T> &ph, const T n[3], T dmean, T r, T ir, T cap,
                                          const T ui[3], const T uj[3], T F[3], unsigned &nlim) {
    const T L = m_log(T(0.5) * r);  // ln(<d>/(2h))
    T a_sq = T(1.5 * PI_D) * ph.mu * dmean * (T(0.25) * r + T(18.0 / 40.0) * L + T(9.0 / 84.0) * L * ir);
    // a_sh (2/(h+<d>))^2 = (pi/2) mu <d> ln(<d>/(2h))
    T a_sh = T(0.5 * PI_D) * ph.mu * dmean * L;
    a_sq = m_max(a_sq, T(0));
    a_sh = m_max(a_sh, T(0));
    if (ph.lub_limiter) {
        if (a_sq > cap) { a_sq = cap; ++nlim; }
        if (a_sh > cap) { a_sh = cap; ++nlim; }
    }
    T upr[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) upr[a] = ui[a] - uj[a];
    const T upn = upr[0] * n[0] + upr[1] * n[1] + upr[2] * n[2];
#pragma unroll
    for (int a = 0; a < 3; ++a) F[a] += -a_sq * upn * n[a] - a_sh * (upr[a] - upn * n[a]);
}

// force and torque on i from one partner (sphere or wall), Sec. 3.1.1 / 3.1.3,
// given m_ij and <d>: contact while overlapping, lubrication on pairs that do
// not overlap, 0 <= h < h_c (in contact the spring-dashpot acts alone, which
// keeps the wet rebound of Sec. 5)
// gap = |x_j - x_i| - (d_i + d_j)/2 (negative: the overlap).
template <typename T>
__device__ __forceinline__ void partner(const PairPar<T> &ph, const T n[3], T gap, const T ui[3], const T wi[3],
                                        T di, const T uj[3], const T wjh[3], T m_ij, T dmean, T F[3], T Tq[3],
                                        unsigned &nlim) {
    const T delta = -gap;
    if (ph.contact && delta > T(0)) contact_force<T>(ph, n, delta, ui, wi, di, uj, wjh, m_ij, T(0.5) * di, F, Tq);
    const T h = gap;
    if (ph.lubrication && h >= T(0) && h < ph.h_c) {
        const T hh = m_max(h, ph.h_min);
        const T q = T(1) / (dmean * hh);  // r and 1/r from one division
        lub_force(ph, n, dmean, dmean * dmean * q, hh * hh * q, m_ij * ph.capfac, ui, uj, F, nlim);
    }
}

// list of particle i: partners j != i with |x_j - x_i| < (d_i+d_j)/2 + extra + skin
// (screened in FP32 with a margin), stored row by row.  Partners within the
// inner shell (range + Phys::shell) fill row i from the front, nlist[i*maxn + k],
// k < nlist_n[i]; the rest fill it from the back, nlist[i*maxn + maxn-1-k],
// k < nlist_o[i].  While no particle of the box has moved more than shell/2
// since the sort, only inner pairs can interact and the substeps leave the
// outer ones alone (BoxDev::moved): with the default skin of half a cell and
// an interaction range of 3 cells the list has 20 partners a particle, the inner
// shell 12.  The FP16-storage form (split = 0) keeps one row, outer partners
// as ~j, and its inner rows apart (k_inner_rows).
// LANES lanes share a particle (the tile's lanes of the particle-side
// kernels): lane l scans the cell rows l, l + LANES, ...
// of the (2R+1)^2 rows around it, counts its partners, takes its offset from
// an exclusive sum over the lanes, then scans again and writes them, so the
// list is in lane-major row order whatever the launch shape.
constexpr int NL_CACHE = 8;  // partners per lane kept between the two passes

#ifndef DPS_NLIST_MINB
#define DPS_NLIST_MINB 4  // 256-thread blocks per SM the register budget is sized for (a latency-bound search)
#endif
__global__ void __launch_bounds__(256, DPS_NLIST_MINB) k_build_nlist(const BoxDev *__restrict__ boxes, const Tile *__restrict__ tiles,
                                                     int ntiles) {
    __shared__ int nl_cache[256][NL_CACHE];
    DPS_FOR_TILES(tiles, ntiles, t) {
        const Tile tl = tiles[t];
        const BoxDev &Bx = boxes[tl.box];
        // lanes per particle of the tile (1 for large boxes, whose lists then
        // run in plain row order; more for boxes with few particles)
        const int LANES = tl.first > 1 ? tl.first : 1;
        const int lane = threadIdx.x % LANES, grp = threadIdx.x / LANES, ngrp = blockDim.x / LANES;
        const Geom g = Bx.g;
        const Phys &ph = Bx.ph;
        const float4 *xf = Bx.xf[0];
        const float reach = (float)(ph.lubrication ? fmax(ph.h_c, 0.0) : 0.0) + SCREEN_MARGIN;
        const float extra = reach + (float)ph.skin, inner = reach + ph.shell;
        const float Lf[3] = {(float)g.n[0], (float)g.n[1], (float)g.n[2]};
        const int R = Bx.R, maxn = Bx.maxn;
        // the trip count is uniform over the block: every lane reaches the shuffles
        for (long long base = tl.begin; base < tl.end; base += ngrp) {
            const long long i = base + grp;
            const bool act = i < tl.end;
            float4 pi = make_float4(0.f, 0.f, 0.f, 0.f);
            int lo[3] = {0, 0, 0}, hi[3] = {-1, -1, -1};
            if (act) {
                pi = xf[i];
                const int b[3] = {containing_cell((double)pi.x, g.n[0]), containing_cell((double)pi.y, g.n[1]),
                                  containing_cell((double)pi.z, g.n[2])};
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    if (g.per[a] && 2 * R + 1 >= g.n[a]) {
                        lo[a] = 0;
                        hi[a] = g.n[a] - 1;
                    } else if (g.per[a]) {
                        lo[a] = b[a] - R;
                        hi[a] = b[a] + R;
                    } else {
                        lo[a] = max(b[a] - R, 0);
                        hi[a] = min(b[a] + R, g.n[a] - 1);
                    }
                }
            }
            const int ny = hi[1] - lo[1] + 1, nz = hi[2] - lo[2] + 1, nrows = act ? ny * nz : 0;
            // the rows, and the x segments of a row (two where it wraps
            // periodically), are visited in ascending cell index of the
            // wrapped cells, so that one lane's partners come out in ascending
            // sorted index (the cells are the sort's keys).  Rows, and row
            // ends, beyond the reach of the particle are left out: of the 9 x 9
            // x 9 cells at a reach of 3.5 cells about half remain, and rows are
            // stepped without divisions (25,000 instructions a warp before;
            // 256^3, eps 0.2: 2.24 -> 1.21 ms).  rm: the largest distance that can be listed, with a
            // margin for the rounding of float positions (boxes below 2^12)
            const float rm = 0.5f * (pi.w + ph.dmax) + extra + SCREEN_MARGIN;
            const bool trim = ph.far_ok != 0, trimx = trim && !(g.per[0] && 2 * R + 1 >= g.n[0]);
            const int roty = lo[1] < 0 ? -lo[1] : (hi[1] > g.n[1] - 1 ? g.n[1] - lo[1] : 0);
            const int rotz = lo[2] < 0 ? -lo[2] : (hi[2] > g.n[2] - 1 ? g.n[2] - lo[2] : 0);
            // distance from coordinate x to the cells [c, c+1) of an axis
            auto away = [&](float x, int c, int ax) {
                float d = fabsf(((float)c + 0.5f) - x);
                if (g.per[ax]) d = fminf(d, fabsf(Lf[ax] - d));
                return fmaxf(d - 0.5f, 0.0f);
            };
            // partners of particle i in this lane's rows r = lane, lane +
            // LANES, ..., in row order, then the sorted order inside a row; the
            // particle ranges of RB rows are loaded together before any is
            // scanned, so their loads are in flight at once
            constexpr int RB = 4;
            auto scan_rows = [&](auto &&fn) {
                int yi = lane, zi = 0;  // row r = yi + ny zi, stepped without divisions
                if (nrows)
                    while (yi >= ny) {
                        yi -= ny;
                        ++zi;
                    }
                while (zi < nz && nrows) {
                    int s[2 * RB], e[2 * RB];
#pragma unroll
                    for (int u = 0; u < RB; ++u) {
                        s[2 * u] = e[2 * u] = s[2 * u + 1] = e[2 * u + 1] = 0;
                        if (zi >= nz) continue;
                        int yy = yi + roty, zz = zi + rotz;
                        yy = lo[1] + (yy >= ny ? yy - ny : yy);
                        zz = lo[2] + (zz >= nz ? zz - nz : zz);
                        yi += LANES;
                        while (yi >= ny) {
                            yi -= ny;
                            ++zi;
                        }
                        int a = lo[0], b = hi[0];
                        if (trim) {
                            const float dy = away(pi.y, yy, 1), dz = away(pi.z, zz, 2);
                            const float h2 = rm * rm - dy * dy - dz * dz;
                            if (!(h2 > 0.0f)) continue;
                            if (trimx) {
                                const float h = sqrtf(h2) + SCREEN_MARGIN;
                                a = max(a, (int)floorf(pi.x - h));
                                b = min(b, (int)floorf(pi.x + h));
                                // a position outside the box or not finite
                                // (the run is flagged): no cells
                                if (a > b || b < 0 || a > g.n[0] - 1) continue;
                            }
                        }
                        const int z = zz < 0 ? zz + g.n[2] : (zz >= g.n[2] ? zz - g.n[2] : zz);
                        const int y = yy < 0 ? yy + g.n[1] : (yy >= g.n[1] ? yy - g.n[1] : yy);
                        const int *cs = Bx.cell_start + cell_index(g, 0, y, z);
                        // [a, b] on the axis, or [0, b'] and [a', n-1] where it wraps
                        const int n0 = g.n[0];
                        const bool wraps = a < 0 || b > n0 - 1;
                        s[2 * u] = cs[wraps ? 0 : a];
                        e[2 * u] = cs[(b > n0 - 1 ? b - n0 : b) + 1];
                        if (wraps) {
                            s[2 * u + 1] = cs[a < 0 ? a + n0 : a];
                            e[2 * u + 1] = cs[n0];
                        }
                    }
#pragma unroll
                    for (int v = 0; v < 2 * RB; ++v)
                        for (int j = s[v]; j < e[v]; ++j) {
                            if (j == i) continue;
                            const float4 pj = xf[j];
                            const float dx = min_image_f(pj.x - pi.x, Lf[0], g.per[0]);
                            const float dy = min_image_f(pj.y - pi.y, Lf[1], g.per[1]);
                            const float dz = min_image_f(pj.z - pi.z, Lf[2], g.per[2]);
                            const float sr = 0.5f * (pi.w + pj.w), d2 = dx * dx + dy * dy + dz * dz;
                            const float rr = sr + extra, ri = sr + inner;
                            if (d2 < rr * rr) fn(j, d2 < ri * ri);
                        }
                }
            };
            // one lane: a single pass writes the list.  Several lanes: pass 1
            // counts and keeps the first NL_CACHE partners of the lane in
            // shared memory (outer ones as ~j); pass 2 writes them (scanning
            // again only past that)
            int *cache = nl_cache[threadIdx.x];
            int *lst = Bx.nlist + i * (long long)maxn;
            const bool split = Bx.split != 0;
            int wi = 0, wo = 0;  // inner and outer partners written
            auto put = [&](int j, bool in) {
                // the callers keep wi + wo below maxn
                lst[split && !in ? maxn - 1 - wo : (split ? wi : wi + wo)] = split || in ? j : ~j;
                wi += in;
                wo += !in;
            };
            auto counts = [&](int ci, int co) {
                if (ci + co > maxn) {
                    atomicOr(Bx.status, ST_NLIST);
                    ci = co = 0;
                }
                Bx.nlist_n[i] = split ? ci : ci + co;
                Bx.nlist_o[i] = split ? co : 0;
            };
            if (LANES == 1) {
                scan_rows([&](int j, bool in) {
                    if (wi + wo < maxn) put(j, in);
                    else (in ? wi : wo)++;
                });
                if (act) counts(wi, wo);
                continue;
            }
            // counts: inner in the low, outer in the high half of a word (a
            // box of several lanes has fewer than 2^15 particles)
            int cnt = 0, cio = 0;
            scan_rows([&](int j, bool in) {
                if (cnt < NL_CACHE) cache[cnt] = in ? j : ~j;
                ++cnt;
                cio += in ? 1 : 0x10000;
            });
            // exclusive sums of the counts over the lanes of the group
            int off = cio;
            for (int o = 1; o < LANES; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, off, o);
                if (lane >= o) off += v;
            }
            const int total = __shfl_sync(0xffffffffu, off, (threadIdx.x & 31) - lane + LANES - 1);
            off -= cio;
            if (!act) continue;
            const int ti = total & 0xffff, to = total >> 16;
            wi = off & 0xffff;
            wo = off >> 16;
            const bool fits = ti + to <= maxn;  // a row that does not stays empty: the run is flagged and stops
            if (cnt <= NL_CACHE) {
                for (int c = 0; c < cnt; ++c) {
                    const int e = cache[c];
                    if (fits) put(e < 0 ? ~e : e, e >= 0);
                }
            } else {
                // (the second scan finds the partners of the first: the bound
                // only keeps a lane inside its own counted slots)
                const int ei = wi + (cio & 0xffff), eo = wo + (cio >> 16);
                scan_rows([&](int j, bool in) {
                    if (fits && (in ? wi < ei : wo < eo)) put(j, in);
                });
            }
            if (lane == 0) counts(ti, to);
        }
    }
}

// the FP64 interaction with sphere j (Sec. 3.1.1 / 3.1.3; separation from the
// FP64 positions): F on particle i, and n x F_t in T (both partners take it
// times their d/2)
__device__ __forceinline__ void pair64_body(const PairPar<double> &pd, const double *__restrict__ xin,
                                            const double *__restrict__ pf, long long cap, const Geom &g, long long j,
                                            const double xi[3], const double ui[3], const double wi[3], double di,
                                            double mi, double rng_extra, double F[3], double T[3], unsigned &nlim) {
    double n[3], uj[3], wjh[3], dx[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) dx[a] = min_image(xin[a * cap + j] - xi[a], g.n[a], g.per[a]);
    const double dist2 = dx[0] * dx[0] + dx[1] * dx[1] + dx[2] * dx[2];
    const double dj = pf[PD * cap + j];
    const double sumr = 0.5 * (di + dj);
    if (!(dist2 > 0.0)) return;
    const double inv = rsqrt(dist2);  // 1/|dx| and |dx| from one reciprocal square root
    const double dist = dist2 * inv;
    if (!(dist < sumr + rng_extra)) return;
    const double mj = pf[PM * cap + j];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        n[a] = dx[a] * inv;
        uj[a] = xin[(3 + a) * cap + j];
    }
    const double A = mi * mj, Bm = mi + mj;           // m_ij = A / Bm
    const double C = 2.0 * di * dj, D = di + dj;      // <d> = C / D
    const double delta = sumr - dist;
    if (pd.contact && delta > 0.0) {
        // the partner's spin only matters in contact (the friction)
#pragma unroll
        for (int a = 0; a < 3; ++a) wjh[a] = 0.5 * dj * xin[(6 + a) * cap + j];
        contact_force(pd, n, delta, ui, wi, di, uj, wjh, A / Bm, 1.0, F, T);
    }
    const double h = dist - sumr;
    if (pd.lubrication && h >= 0.0 && h < pd.h_c) {
        // one division for m_ij, <d>, r = <d>/hh and 1/r
        const double hh = fmax(h, pd.h_min);
        const double q = 1.0 / (Bm * D * hh * C);
        const double r = C * C * Bm * q;                // <d> / hh
        const double ir = Bm * D * D * hh * hh * q;     // hh / <d>
        lub_force(pd, n, C * C * Bm * hh * q, r, ir, A * D * hh * C * q * pd.capfac, ui, uj, F, nlim);
    }
}
// the mixed forms' pair within H_NEAR of contact.  The float copies of the
// positions carry absolute errors of up to ~3e-5 at x ~ 256, too coarse for
// such gaps, so the separation comes from the FP64 positions: |dx|^2 - s^2
// in FP64, divided by |dx| + s in FP32, a gap (or overlap) with FP32's
// relative precision however small it is; the forces then run in FP32 like
// every other pair.  Out of line, and returning its terms, so that the rare
// call costs the FP32 pair loop no registers.
struct NearTerms {
    float F[3], T[3];
    unsigned nlim;
};
__device__ __noinline__ NearTerms near_pair32(const BoxDev &Bx, const double *__restrict__ xin,
                                              const float4 *__restrict__ vin, const float4 *__restrict__ oin,
                                              const PairPar<float> &pfl, long long i, int j, float4 pi, float4 pj,
                                              float4 vi, float4 oi, float rng_extra_f) {
    NearTerms o = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}, 0u};
    const double *pf = Bx.pf[Bx.cur];
    const long long cap = Bx.cap;
    const Geom g = Bx.g;
    double dx[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) dx[a] = min_image(xin[a * cap + j] - xin[a * cap + i], g.n[a], g.per[a]);
    const double d2 = dx[0] * dx[0] + dx[1] * dx[1] + dx[2] * dx[2];
    const double s = 0.5 * (pf[PD * cap + i] + pf[PD * cap + j]);
    const float distf = sqrtf((float)d2);
    if (!(distf > 0.f)) return o;
    const float gap = (float)fma(-s, s, d2) / (distf + (float)s);
    if (!(gap < rng_extra_f)) return o;
    const float4 vj = vin[j], oj = oin[j];
    const float inv = 1.0f / distf;
    const float n[3] = {(float)dx[0] * inv, (float)dx[1] * inv, (float)dx[2] * inv};
    const float uif[3] = {vi.x, vi.y, vi.z}, wif[3] = {oi.x, oi.y, oi.z};
    const float uj[3] = {vj.x, vj.y, vj.z};
    const float wjh[3] = {0.5f * pj.w * oj.x, 0.5f * pj.w * oj.y, 0.5f * pj.w * oj.z};
    const float m_ij = vi.w * vj.w / (vi.w + vj.w);
    const float dmean = 2.0f * pi.w * pj.w / (pi.w + pj.w);
    partner<float>(pfl, n, gap, uif, wif, pi.w, uj, wjh, m_ij, dmean, o.F, o.T, o.nlim);
    return o;
}

// contact or lubrication with face `side` of axis a, in FP64 (out of line: few
// particles of few warps need it)
__device__ __noinline__ void wall_exact(const BoxDev &Bx, long long i, int a, int side, double xa, const double ui[3],
                                        const double wi[3], double F[3], double T[3]) {
    const Phys &ph = Bx.ph;
    const double *pf = Bx.pf[Bx.cur];
    const double di = pf[PD * Bx.cap + i], mi = pf[PM * Bx.cap + i];
    const double dist = side == 0 ? xa : Bx.g.n[a] - xa;
    if (!(dist < 0.5 * di + (ph.lubrication ? fmax(ph.h_c, 0.0) : 0.0))) return;
    const PairPar<double> pd = pair_par<double>(ph);
    const double zero[3] = {0, 0, 0}, s = side == 0 ? -1.0 : 1.0;
    const double n[3] = {a == 0 ? s : 0.0, a == 1 ? s : 0.0, a == 2 ? s : 0.0};
    unsigned nlim = 0;
    partner<double>(pd, n, dist - 0.5 * di, ui, wi, di, zero, zero, mi, 2.0 * di, F, T, nlim);
    if (nlim) atomicAdd(&Bx.counters[CNT_LUB_LIMITED], (unsigned long long)nlim);
}

// the rare branches of the update: a position off a periodic axis, the exact
// displacement, the linked cell after the last substep
__device__ __forceinline__ double fold_axis(double xn, int n) {
    const double L = n;
    if (xn >= L) xn -= L;
    else if (xn < 0.0) xn += L;
    if (xn >= L || xn < 0.0) xn -= L * floor(xn / L);
    if (xn >= L) xn -= L;
    return xn;
}
__device__ __forceinline__ void check_skin(const BoxDev &Bx, long long i, double x, double y, double z) {
    const double *xs = Bx.pf[Bx.cur] + PXS0 * Bx.cap + i;
    const double xn3[3] = {x, y, z};
    double d2 = 0.0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double dd = min_image(xn3[a] - xs[a * Bx.cap], Bx.g.n[a], Bx.g.per[a]);
        d2 += dd * dd;
    }
    if (d2 > Bx.ph.skin_half2) atomicOr(Bx.status, ST_SKIN);
    if (!(d2 < 1e30)) atomicOr(Bx.status, ST_NAN);
}
__device__ __forceinline__ int new_cell(const BoxDev &Bx, double x, double y, double z) {
    return (int)particle_cell(Bx.g, x, y, z, Bx.status);
}
// out of line in boxes without walls, where occupancy counts (a box with walls
// calls the wall contact already): with FP64 comparisons and conversions gone
// and 5 -> 7 blocks per SM the DEM of 101x90x77 at eps 0.36 took 6.5 -> 6.2 ms a
// step, and the update of the mixed forms with 3 -> 4 blocks 11.7 -> 11.0 ms
// (192^3, eps 0.38, FP32) and 9.7 -> 8.8 ms (32^3)
__device__ __noinline__ double fold_axis_call(double xn, int n) { return fold_axis(xn, n); }
__device__ __noinline__ void check_skin_call(const BoxDev &Bx, long long i, double x, double y, double z) {
    check_skin(Bx, i, x, y, z);
}
__device__ __noinline__ int new_cell_call(const BoxDev &Bx, double x, double y, double z) { return new_cell(Bx, x, y, z); }

// one thread per particle: wall partners (WALLS), then Eq. particle_motion
// (semi-implicit Euler) and the outputs of the substep.  Comparisons and
// conversions are integer or FP32 operations (an FP64 compare or conversion
// costs as much as an FP64 multiply-add), and the spin is integrated only
// under a torque: 10 FP64 instructions for a particle away from walls, where
// ~55 were issued before.
template <bool WALLS, bool F64>
__device__ __forceinline__ void finish_particle(const BoxDev &Bx, long long i, int src_tmp, double F[3], double T[3],
                                               int key_out, int *moved_out) {
    const double *xin = src_tmp ? Bx.xtmp : Bx.pf[Bx.cur];
    double *xout = src_tmp ? Bx.pf[Bx.cur] : Bx.xtmp;
    const double *pf = Bx.pf[Bx.cur];
    const long long cap = Bx.cap;
    const Geom &g = Bx.g;
    const Phys &ph = Bx.ph;
    double xi[3], ui[3], wi[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        xi[a] = xin[a * cap + i];
        ui[a] = xin[(3 + a) * cap + i];
        wi[a] = xin[(6 + a) * cap + i];
    }
    const float4 xs = Bx.xs[i];  // position at the last sort, and d
    // walls: the faces of every non-periodic axis (m_ij = m_i, <d> = 2 d_i),
    // screened in FP32 (xs carries d) with the margin of the pair screen.  The
    // FP64 form takes the lubrication from the integer path (fx_wall) and
    // leaves contact to the FP64 body out of line: inlined, six faces' worth of
    // FP64 cost 211 registers a thread (closures with walls, 75 x 61 x 90: DEM
    // substep 67 -> 55 us with three blocks per SM, 64 with one)
    if (WALLS && !(g.per[0] && g.per[1] && g.per[2])) {
        const float reach = 0.5f * xs.w + (float)(ph.lubrication ? fmax(ph.h_c, 0.0) : 0.0) + SCREEN_MARGIN;
        const float fx3[3] = {to_float(xi[0]), to_float(xi[1]), to_float(xi[2])};
#pragma unroll 1
        for (int f = 0; f < 6; ++f) {
            const int a = f >> 1, side = f & 1;
            const float xf = a == 0 ? fx3[0] : (a == 1 ? fx3[1] : fx3[2]);
            const int n_a = a == 0 ? g.n[0] : (a == 1 ? g.n[1] : g.n[2]);
            const int per = a == 0 ? g.per[0] : (a == 1 ? g.per[1] : g.per[2]);
            const float away = side ? (float)n_a - xf : xf;
            if (per || (!(away < reach) && ph.far_ok)) continue;
            const double xa = a == 0 ? xi[0] : (a == 1 ? xi[1] : xi[2]);
            int kind = FX_EXACT;
            if (F64 && ph.fx.ok && ph.lubrication) {
                const DemPart q = Bx.part[Bx.cur][i];
                double al, be;
                kind = fx_wall(fma(-0.5, pf[PD * cap + i], side ? n_a - xa : xa), (u64)q.inv_d, ph.h_c, ph.h_min,
                               ph.fx, al, be);
                if (kind == FX_LUB) {
                    const float capf = (float)ph.capfac * 0.999f;
                    if (ph.lub_limiter && !(fx_approx(be) * q.imf < capf && fx_approx(al) * q.imf < capf)) {
                        const double lim = pf[PM * cap + i] * ph.capfac;
                        const unsigned nlim = (be > lim) + (al > lim);
                        be = be > lim ? lim : be;
                        al = al > lim ? lim : al;
                        if (nlim) atomicAdd(&Bx.counters[CNT_LUB_LIMITED], (unsigned long long)nlim);
                    }
#pragma unroll
                    for (int k = 0; k < 3; ++k) F[k] -= (k == a ? be : al) * ui[k];
                }
            }
            if (kind == FX_EXACT) wall_exact(Bx, i, a, side, xa, ui, wi, F, T);
        }
    }
    // Eq. particle_motion, semi-implicit Euler with I = m d^2 / 10
    const double dt_m = ph.dt_dem * pf[PIM * cap + i];
    double xn3[3], un3[3], wn3[3] = {wi[0], wi[1], wi[2]};
    if ((fx_bits(T[0]) | fx_bits(T[1]) | fx_bits(T[2])) << 1) {  // (either zero shifts out its sign)
        const double dt_I = ph.dt_dem * pf[PII * cap + i];
#pragma unroll
        for (int a = 0; a < 3; ++a) wn3[a] = wi[a] + dt_I * T[a];
    }
    float xf[3], d2f = 0.0f;
    const float xsf[3] = {xs.x, xs.y, xs.z};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double Ft = pf[(PFH0 + a) * cap + i] + F[a];
        const double un = ui[a] + dt_m * Ft;
        double xn = xi[a] + ph.dt_dem * un;
        if (g.per[a]) {
            // a particle that left the box folds back in; 0 <= xn < L compared
            // as integers (the order of the bits is that of the values)
            if (!(fx_bits(xn) < ph.Lbits[a])) xn = WALLS ? fold_axis(xn, g.n[a]) : fold_axis_call(xn, g.n[a]);
        }
        xn3[a] = xn;
        un3[a] = un;
        xout[a * cap + i] = xn;
        xout[(3 + a) * cap + i] = un;
        xout[(6 + a) * cap + i] = wn3[a];
        xf[a] = to_float(xn);
        const float dd = min_image_f(xf[a] - xsf[a], (float)g.n[a], g.per[a]);
        d2f += dd * dd;
    }
    Bx.xf[1 - src_tmp][i] = make_float4(xf[0], xf[1], xf[2], xs.w);
    if (F64) {
        DemRec r;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            r.x[a] = fx_from(xn3[a], ph.fx.frac);
            r.u[a] = un3[a];
        }
        Bx.rec[1 - src_tmp][i] = r;
    } else {
        const float mf = Bx.vf[src_tmp][i].w;
        Bx.vf[1 - src_tmp][i] = make_float4(to_float(un3[0]), to_float(un3[1]), to_float(un3[2]), mf);
        Bx.of[1 - src_tmp][i] = make_float4(to_float(wn3[0]), to_float(wn3[1]), to_float(wn3[2]), 0.f);
    }
    if (key_out) {
        // last substep of the subcycle: the linked cell of the new position,
        // counted for the sort that follows (its counting pass)
        const int c = WALLS ? new_cell(Bx, xn3[0], xn3[1], xn3[2]) : new_cell_call(Bx, xn3[0], xn3[1], xn3[2]);
        Bx.key[i] = c;
        atomicAdd(&Bx.count[c], 1);
    }
    // moved beyond skin/2 since the sort, or not finite: decided in FP32
    // where its rounding cannot matter, else in FP64
    if (!(d2f < ph.shell_near2)) *moved_out = 1;
    if (!(d2f < ph.skin_near2)) {
        if (WALLS) check_skin(Bx, i, xn3[0], xn3[1], xn3[2]);
        else check_skin_call(Bx, i, xn3[0], xn3[1], xn3[2]);
    }
}

// ---- the substep of the mixed forms ----------------------------------------------------
// src_tmp = 0: read x/u/w (and the float positions) from the current set,
// write the ping-pong buffers; src_tmp = 1: the other way round.
// k_dem_pairsum_mixed: lane groups of LANES lanes per particle walk its list;
// pairs away from contact run in FP32 from the float copies, pairs near
// contact in FP32 from an FP64 separation (out of line); the group's sums (a
// fixed xor tree) go
// to psum[6][cap] (force, torque) and the lubrication-cap count to the
// counters.  k_dem_integrate then adds the walls and integrates, one thread
// per particle.  Two kernels so that each has its own register budget: the
// pair loop waits on the partners' loads and needs every warp slot of the SM,
// the FP64 update needs registers.
#ifndef DPS_INTEG_MINB
#define DPS_INTEG_MINB 4  // 128-thread blocks per SM the register budget of the update is sized for
#endif
#ifndef DPS_MIXED_MINB
#define DPS_MIXED_MINB 4  // 256-thread blocks per SM the register budget of the pair loop is sized for
#endif
template <int LANES, typename Sink>
__device__ __forceinline__ void pairsum_tile(const BoxDev &Bx, const Tile &tl, int src_tmp, int outer, Sink &&sink) {
    const int lane = threadIdx.x % LANES, grp = threadIdx.x / LANES, ngrp = blockDim.x / LANES;
    {
        const double *xin = src_tmp ? Bx.xtmp : Bx.pf[Bx.cur];
        const float4 *fin = Bx.xf[src_tmp], *vin = Bx.vf[src_tmp], *oin = Bx.of[src_tmp];
        const Geom g = Bx.g;
        const Phys &ph = Bx.ph;
        const float rng_extra_f = (float)(ph.lubrication ? fmax(ph.h_c, 0.0) : 0.0);
        const float Lf[3] = {(float)g.n[0], (float)g.n[1], (float)g.n[2]};
        const PairPar<float> pfl = pair_par<float>(ph);
        const long long cap = Bx.cap;
        // the trip count is uniform over the block, so every lane reaches the shuffles
        for (long long base = tl.begin; base < tl.end; base += ngrp) {
            const long long i = base + grp;
            const bool act = i < tl.end;
            float Ff[3] = {0, 0, 0}, Tf[3] = {0, 0, 0};
            unsigned nlim = 0;
            if (act) {
                const float4 pi = fin[i], vi = vin[i], oi = oin[i];
                const int *row = Bx.nlist + i * (long long)Bx.maxn;
                int ni = Bx.nlist_n[i], nn = ni + (outer ? Bx.nlist_o[i] : 0);
                if (!Bx.split && !outer) {
                    row = Bx.ilist + i * (long long)Bx.maxi;
                    ni = nn = Bx.ilist_n[i];
                }
                const int back = Bx.maxn - 1 + ni;  // outer partner k - ni sits at maxn-1 - (k - ni)
                for (int k = lane; k < nn; k += LANES) {
                    int j = row[k < ni ? k : back - k];
                    if (j < 0) {  // (one-row form) an outer partner, or a gap of the inner rows
                        if (!outer) continue;
                        j = ~j;
                    }
                    const float4 pj = fin[j];
                    const float fx = min_image_f(pj.x - pi.x, Lf[0], g.per[0]);
                    const float fy = min_image_f(pj.y - pi.y, Lf[1], g.per[1]);
                    const float fz = min_image_f(pj.z - pi.z, Lf[2], g.per[2]);
                    const float sumr_f = 0.5f * (pi.w + pj.w);
                    const float fr = sumr_f + rng_extra_f + SCREEN_MARGIN;
                    const float d2f = fx * fx + fy * fy + fz * fz;
                    if (!(d2f < fr * fr)) continue;
                    const float distf = sqrtf(d2f);
                    if (distf - sumr_f > (float)H_NEAR + SCREEN_MARGIN) {
                        // away from contact: the separation from the float copies
                        if (!(distf < sumr_f + rng_extra_f)) continue;
                        const float4 vj = vin[j], oj = oin[j];
                        const float inv = 1.0f / distf;
                        const float n[3] = {fx * inv, fy * inv, fz * inv};
                        const float uif[3] = {vi.x, vi.y, vi.z}, wif[3] = {oi.x, oi.y, oi.z};
                        const float uj[3] = {vj.x, vj.y, vj.z};
                        const float wjh[3] = {0.5f * pj.w * oj.x, 0.5f * pj.w * oj.y, 0.5f * pj.w * oj.z};
                        const float m_ij = vi.w * vj.w / (vi.w + vj.w);
                        const float dmean = 2.0f * pi.w * pj.w / (pi.w + pj.w);
                        partner<float>(pfl, n, distf - sumr_f, uif, wif, pi.w, uj, wjh, m_ij, dmean, Ff, Tf, nlim);
                        continue;
                    }
                    // near contact: the separation from the FP64 positions
                    const NearTerms o = near_pair32(Bx, xin, vin, oin, pfl, i, j, pi, pj, vi, oi, rng_extra_f);
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        Ff[a] += o.F[a];
                        Tf[a] += o.T[a];
                    }
                    nlim += o.nlim;
                }
            }
            if (LANES > 1) {
#pragma unroll
                for (int o = LANES / 2; o > 0; o >>= 1) {
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        Ff[a] += __shfl_xor_sync(0xffffffffu, Ff[a], o);
                        Tf[a] += __shfl_xor_sync(0xffffffffu, Tf[a], o);
                    }
                    nlim += __shfl_xor_sync(0xffffffffu, nlim, o);
                }
            }
            if (act && lane == 0) {
                sink(i, Ff, Tf);
                if (nlim) atomicAdd(&Bx.counters[CNT_LUB_LIMITED], (unsigned long long)nlim);
            }
        }
    }
}

// LANES 0: boxes of several lane classes in one launch, each tile with its own
// (a batch launched once per class and substep before: 12 boxes, FP32, DEM 2.8 ->
// 2.5 ms a step)
template <int LANES>
__global__ void __launch_bounds__(256, DPS_MIXED_MINB) k_dem_pairsum_mixed(const BoxDev *__restrict__ boxes,
                                                                       const Tile *__restrict__ tiles, int ntiles,
                                                                       int src_tmp) {
    DPS_FOR_TILES(tiles, ntiles, t) {
        const Tile tl = tiles[t];
        const BoxDev &Bx = boxes[tl.box];
        const long long cap = Bx.cap;
        auto store = [&](long long i, const float Ff[3], const float Tf[3]) {
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                Bx.psum[a * cap + i] = (double)Ff[a];
                Bx.psum[(3 + a) * cap + i] = (double)Tf[a];
            }
        };
        // outer partners only once a particle of the box has moved shell/2
        const int outer = Bx.moved[src_tmp];
        // cleared for this substep's update to set, by one thread of the box: a
        // store from every block to the word all blocks read costs 20 us a launch
        if (tl.begin == 0 && threadIdx.x == 0) Bx.moved[1 - src_tmp] = 0;
        if (LANES > 0) {
            pairsum_tile<LANES ? LANES : 1>(Bx, tl, src_tmp, outer, store);
        } else {
            switch (Bx.dem_lanes) {
                case 8: pairsum_tile<8>(Bx, tl, src_tmp, outer, store); break;
                case 4: pairsum_tile<4>(Bx, tl, src_tmp, outer, store); break;
                case 2: pairsum_tile<2>(Bx, tl, src_tmp, outer, store); break;
                default: pairsum_tile<1>(Bx, tl, src_tmp, outer, store);
            }
        }
    }
}

// Few particles (tiles of at most 32, 8 lanes each, which fill the chip once): a
// block sums the pairs of its tile, passes the sums through shared memory, and
// its first warp updates the 32 particles: one launch a substep, and no trip of
// the sums through global memory (18.8k spheres in 32^3: 17.6 -> 16.5 us a
// substep).  The blocks of a substep read slot sd
// mod 3 of Bx.moved, set the next and clear the one after it, which the
// substep before this one read: no slot is read and written in one launch.
// A tile that is its whole box (solo) takes all n substeps from sd in one
// launch.
#ifndef DPS_MIXED8_MINB
#define DPS_MIXED8_MINB 4  // one wave of the largest count (3 blocks: 16.5 -> 19 us)
#endif
template <bool WALLS>
__global__ void __launch_bounds__(256, DPS_MIXED8_MINB) k_dem_mixed8(const BoxDev *__restrict__ boxes,
                                                                     const Tile *__restrict__ tiles, int sd, int n,
                                                                     int n_dem) {
    __shared__ float sums[6][32];
    const Tile tl = tiles[blockIdx.x];
    const BoxDev &Bx = boxes[tl.box];
    auto store = [&](long long i, const float Ff[3], const float Tf[3]) {
        const int k = (int)(i - tl.begin);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            sums[a][k] = Ff[a];
            sums[3 + a][k] = Tf[a];
        }
    };
#pragma unroll 1
    for (int q = 0; q < n; ++q, ++sd) {
        const int src_tmp = sd & 1, slot = sd % 3;
        const int outer = Bx.moved[slot];
        if (tl.begin == 0 && threadIdx.x == 0) Bx.moved[slot == 0 ? 2 : slot - 1] = 0;
        pairsum_tile<8>(Bx, tl, src_tmp, outer, store);
        __syncthreads();
        const long long i = tl.begin + threadIdx.x;
        if (threadIdx.x < 32 && i < tl.end) {
            double F[3], T[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                F[a] = (double)sums[a][threadIdx.x];
                T[a] = (double)sums[3 + a][threadIdx.x];
            }
            finish_particle<WALLS, false>(Bx, i, src_tmp, F, T, sd == n_dem - 1, Bx.moved + (slot == 2 ? 0 : slot + 1));
        }
        if (q + 1 < n) __syncthreads();
    }
}

// walls and Eq. particle_motion of the mixed forms, one thread per particle
template <bool WALLS>
__global__ void __launch_bounds__(128, DPS_INTEG_MINB) k_dem_integrate(const BoxDev *__restrict__ boxes,
                                                                     const Tile *__restrict__ tiles, int ntiles,
                                                                     int src_tmp, int key_out) {
    DPS_FOR_TILES(tiles, ntiles, t) {
        const Tile tl = tiles[t];
        const BoxDev &Bx = boxes[tl.box];
        const long long cap = Bx.cap;
        for (long long i = tl.begin + threadIdx.x; i < tl.end; i += blockDim.x) {
            double F[3], T[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                F[a] = Bx.psum[a * cap + i];
                T[a] = Bx.psum[(3 + a) * cap + i];
            }
            finish_particle<WALLS, false>(Bx, i, src_tmp, F, T, key_out, Bx.moved + 1 - src_tmp);
        }
    }
}

// The inner rows of the FP16-storage form: the inner partners of row i, each kept by
// the lane (position in the full row modulo the box's lanes per particle) and
// in the order that the full row gives it, so that a substep over the inner
// rows adds in the same order as one over the full rows.  Lanes with fewer
// inner partners end in gaps (-1).  (A change in the last bit of a force, far
// inside the FP32 forms' tolerance, flips roundings of the FP16 populations:
// 1e-3 of a force after a few steps.)
__global__ void __launch_bounds__(128) k_inner_rows(const BoxDev *__restrict__ boxes, const Tile *__restrict__ tiles,
                                                    int ntiles) {
    DPS_FOR_TILES(tiles, ntiles, t) {
        const Tile tl = tiles[t];
        const BoxDev &Bx = boxes[tl.box];
        const int lanes = Bx.dem_lanes;
        for (long long i = tl.begin + threadIdx.x; i < tl.end; i += blockDim.x) {
            const int n = Bx.nlist_n[i];
            const int *row = Bx.nlist + i * (long long)Bx.maxn;
            int *out = Bx.ilist + i * (long long)Bx.maxi;
            int used[8] = {0, 0, 0, 0, 0, 0, 0, 0}, rows = 0;
            for (int k0 = 0; k0 < n; k0 += lanes)
#pragma unroll
                for (int l = 0; l < 8; ++l)
                    if (l < lanes && k0 + l < n && row[k0 + l] >= 0) out[used[l]++ * lanes + l] = row[k0 + l];
#pragma unroll
            for (int l = 0; l < 8; ++l) rows = max(rows, used[l]);
#pragma unroll
            for (int l = 0; l < 8; ++l)
                if (l < lanes)
                    for (int m = used[l]; m < rows; ++m) out[m * lanes + l] = -1;
            Bx.ilist_n[i] = rows * lanes;
        }
    }
}

// block-wide exclusive sum of one int per thread (blockDim a multiple of 32,
// at most 256); total over the block; ws: 9 ints of shared memory
__device__ __forceinline__ int block_excl_sum(int v, int *ws, int &total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += u;
    }
    if (lane == 31) ws[wid] = inc;
    __syncthreads();
    if (threadIdx.x < 32) {
        const int w = lane < nw ? ws[lane] : 0;
        int wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += u;
        }
        if (lane < nw) ws[lane] = wi - w;
        if (lane == nw - 1) ws[8] = wi;
    }
    __syncthreads();
    const int r = ws[wid] + inc - v;
    total = ws[8];
    __syncthreads();  // ws may be reused
    return r;
}

// ---- FP64 form: every pair once (Newton's third law) ------------------------------
// The FP64 pair chain is what bounds this form on GB300 (a dense settling box
// keeps the FP64 pipe ~70 % busy), and the contact and lubrication laws of
// Sec. 3.1.1 / 3.1.3 are antisymmetric: F_ji = -F_ij, and with n_ji = -n_ij,
// F_t,ji = -F_t,ij the torques (d/2) n x F_t of both partners share n x F_t.
// So each substep evaluates each pair of the neighbour list once and a second
// kernel gathers, per particle and in a fixed order (its own pairs by
// ascending partner, then the pairs owned by its lower partners by ascending
// owner, then the walls), before the explicit update of Eq. particle_motion.

// After the list build: the pairs particle i owns (partners j > i) get
// consecutive slots from a per-block allocation, inner ones first (hoff, hn),
// outer ones (hoff2, hn2) behind the inner slots of the block, each by ascending
// j; its partners k < i go to rrow (inner, then outer, ascending k) until
// k_reverse_slots replaces them by the slots of the pairs (k, i).  Ranks by
// counting keep the rows free of any sort.
__global__ void __launch_bounds__(256) k_half_rows(const BoxDev *__restrict__ boxes, const Tile *__restrict__ tiles,
                                                   int ntiles) {
    __shared__ int ws[9];
    __shared__ unsigned long long sbase;
    DPS_FOR_TILES(tiles, ntiles, t) {
        const Tile tl = tiles[t];
        const BoxDev &Bx = boxes[tl.box];
        const int maxn = Bx.maxn;
        for (long long base = tl.begin; base < tl.end; base += blockDim.x) {  // uniform trip count
            const long long i = base + threadIdx.x;
            const bool act = i < tl.end;
            // part 0: the inner partners (row from the front), part 1: the
            // outer ones (from the back)
            int nn[2] = {0, 0}, nh[2] = {0, 0}, off[2], total[2];
            const int *row[2] = {Bx.nlist, Bx.nlist};
            if (act) {
                nn[0] = Bx.nlist_n[i];
                nn[1] = Bx.nlist_o[i];
                row[0] = Bx.nlist + i * (long long)maxn;
                row[1] = row[0] + maxn - 1;
                for (int k = 0; k < nn[0]; ++k) nh[0] += row[0][k] > i;
                for (int k = 0; k < nn[1]; ++k) nh[1] += row[1][-k] > i;
            }
            off[0] = block_excl_sum(nh[0], ws, total[0]);
            off[1] = block_excl_sum(nh[1], ws, total[1]) + total[0];
            if (threadIdx.x == 0) sbase = atomicAdd(Bx.ptop, (unsigned long long)(total[0] + total[1]));
            __syncthreads();
            const long long sb = (long long)sbase;
            __syncthreads();  // sbase is written again in the next round
            if (!act) continue;
            if (sb + total[0] + total[1] > Bx.pcap) {  // not reached: pcap bounds the pairs of any list
                atomicOr(Bx.status, ST_NLIST);
                Bx.hn[i] = Bx.rn[i] = Bx.hn2[i] = Bx.rn2[i] = 0;
                continue;
            }
            Bx.hoff[i] = (int)(sb + off[0]);
            Bx.hoff2[i] = (int)(sb + off[1]);
            Bx.hn[i] = nh[0];
            Bx.hn2[i] = nh[1];
            Bx.rn[i] = nn[0] - nh[0];
            Bx.rn2[i] = nn[1] - nh[1];
            int *rr = Bx.rrow + i * (long long)maxn;
            const unsigned char me = (unsigned char)((i - tl.begin) & 31);
#pragma unroll
            for (int w = 0; w < 2; ++w) {
                const long long h0 = sb + off[w];
                const int n = nn[w], st = w ? -1 : 1;
                const int *r0 = row[w];
                bool asc = true;  // rows of one lane come out ascending
                for (int k = 1; k < n; ++k) asc = asc && r0[st * k] > r0[st * (k - 1)];
                if (asc) {
                    const int lo = n - nh[w];
                    for (int k = 0; k < lo; ++k) rr[k] = r0[st * k];
                    for (int k = lo; k < n; ++k) {
                        Bx.hj[h0 + k - lo] = r0[st * k];
                        Bx.hl[h0 + k - lo] = me;
                    }
                } else {
                    for (int k = 0; k < n; ++k) {
                        const int j = r0[st * k];
                        const bool up = j > i;
                        int r = 0;  // rank of j among the partners on its side of i
                        for (int m = 0; m < n; ++m) {
                            const int o = r0[st * m];
                            r += o < j && (up ? o > i : o < i);
                        }
                        if (up) {
                            Bx.hj[h0 + r] = j;
                            Bx.hl[h0 + r] = me;
                        } else {
                            rr[r] = j;
                        }
                    }
                }
                rr += n - nh[w];
            }
        }
    }
}

// rrow: lower partner k -> the slot of the pair (k, i) (binary search of i in
// the ascending row of k)
__global__ void __launch_bounds__(256) k_reverse_slots(const BoxDev *__restrict__ boxes,
                                                       const Tile *__restrict__ tiles, int ntiles) {
    DPS_FOR_TILES(tiles, ntiles, t) {
        const Tile tl = tiles[t];
        const BoxDev &Bx = boxes[tl.box];
        for (long long i = tl.begin + threadIdx.x; i < tl.end; i += blockDim.x) {
            const int ni = Bx.rn[i], nr = ni + Bx.rn2[i];
            int *rr = Bx.rrow + i * (long long)Bx.maxn;
            for (int r = 0; r < nr; ++r) {
                const int k = rr[r];
                const int hk = r < ni ? Bx.hn[k] : Bx.hn2[k], ok = r < ni ? Bx.hoff[k] : Bx.hoff2[k];
                const int *h = Bx.hj + ok;
                int lo = 0, hi = hk;
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (h[mid] < i)
                        lo = mid + 1;
                    else
                        hi = mid;
                }
                if (lo < hk && h[lo] == i) {
                    rr[r] = ok + lo;
                } else {  // not reached: the list search is symmetric
                    rr[r] = -1;
                    atomicOr(Bx.status, ST_NLIST);
                }
            }
        }
    }
}

// The pairs of a substep.  A warp takes chunks of 32 particles of a tile: their
// owned pairs lie in consecutive slots (k_half_rows), which the lanes screen in
// FP32 (with a margin) 32 at a time.  Pairs that pass go to a queue of the warp
// and are evaluated 32 at a time, one per lane: separation, gap, logarithm and
// reciprocal of a lubrication pair in 64-bit integers (fx_pair), its force in
// 14 FP64 operations.  Pairs that overlap (or leave the range of that path) go to
// a queue of the block, evaluated together by the exact FP64 contact /
// lubrication body at the end of the tile, so that few warps pay for it (an FP64
// instruction costs a warp the same whatever number of its lanes are active).
// Every owned slot gets its flag; the result of a slot depends on its pair alone.
// The FP64 body for every pair took ~120 FP64 warp instructions of ~19 cycles
// per 32 pairs (70 % of the FP64 pipe).  DEM substep (this kernel and the
// gather) before / after, FP64: 256^3, eps 0.2, d 1.5: 4.34 / 2.02 ms; 101 x 90
// x 77, eps 0.36 with contacts: 1.13 / 0.48 ms.  At 128^3 this kernel takes
// 140 us: 1100 instructions per 32 pairs, FP64 pipe 35 %.
constexpr int PAIR_WARPS = 4;
constexpr int EXACT_CAP = 512;  // queued pairs of a tile; past it a pair is evaluated at once

struct PairQueue {
    int slot[PAIR_WARPS][64], j[PAIR_WARPS][64], i[PAIR_WARPS][64];  // rings, one per warp
    int eslot[EXACT_CAP], ej[EXACT_CAP], ei[EXACT_CAP], en;
};

// m_ij capfac and its reciprocal's FP64 Newton steps (x = 1/m_i + 1/m_j)
__device__ __forceinline__ double fx_recip(double x, float xf) {
    double y = (double)__fdividef(1.0f, xf);
    y = fma(y, fma(-x, y, 1.0), y);
    return fma(y, fma(-x, y, 1.0), y);
}

#ifndef DPS_PAIRS_MINB
#define DPS_PAIRS_MINB 7  // 128-thread blocks per SM the register budget is sized for
#endif
// the pairs of one tile (Qs.en is 0 before and after; ends with a barrier)
__device__ __forceinline__ void pairs64_tile(const BoxDev &Bx, const Tile &tl, int src_tmp, PairQueue &Qs) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    {
        const double *xin = src_tmp ? Bx.xtmp : Bx.pf[Bx.cur];
        const float4 *fin = Bx.xf[src_tmp];
        const DemRec *rec = Bx.rec[src_tmp];
        const DemPart *part = Bx.part[Bx.cur];
        const double *pf = Bx.pf[Bx.cur];
        const long long cap = Bx.cap;
        const Geom &g = Bx.g;
        const Phys &ph = Bx.ph;
        const double rng_extra = ph.lubrication ? fmax(ph.h_c, 0.0) : 0.0;
        const float rng_extra_f = (float)rng_extra;
        const float Lf[3] = {(float)g.n[0], (float)g.n[1], (float)g.n[2]};
        const PairPar<double> pd = pair_par<double>(ph);
        const bool fx = ph.fx.ok != 0;
        const float capf = (float)ph.capfac * 0.999f;
        unsigned nlim = 0;

        // the FP64 body of slot sl, the pair (i, j)
        auto exact = [&](int sl, int i, int j) {
            double xi[3], ui[3], wi[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                xi[a] = xin[a * cap + i];
                ui[a] = xin[(3 + a) * cap + i];
                wi[a] = xin[(6 + a) * cap + i];
            }
            double Fq[3] = {0, 0, 0}, Cq[3] = {0, 0, 0};
            pair64_body(pd, xin, pf, cap, g, j, xi, ui, wi, pf[PD * cap + i], pf[PM * cap + i], rng_extra, Fq, Cq,
                        nlim);
            // n x F_t, nonzero only for pairs in contact with friction, in a
            // plane of its own, flagged 2
            const long long sq = sl;
            PairRes r = {{Fq[0], Fq[1], Fq[2]}, 1};
            if (Cq[0] != 0.0 || Cq[1] != 0.0 || Cq[2] != 0.0) {
#pragma unroll
                for (int a = 0; a < 3; ++a) Bx.ptan[3 * sq + a] = Cq[a];
                r.flag = 2;
            }
            Bx.pres[sq] = r;
        };
        // entry k of the warp's queue
        auto eval = [&](int k) {
            const int sl = Qs.slot[wid][k & 63], i = Qs.i[wid][k & 63], j = Qs.j[wid][k & 63];
            int kind = FX_EXACT;
            if (fx) {
                const DemRec ri = rec[i], rj = rec[j];
                const DemPart pi = part[i], pj = part[j];
                i64 dx[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    dx[a] = rj.x[a] - ri.x[a];
                    if (g.per[a]) {
                        const i64 L = (i64)g.n[a] << ph.fx.frac, h = L >> 1;
                        dx[a] = dx[a] > h ? dx[a] - L : (dx[a] < -h ? dx[a] + L : dx[a]);
                    }
                }
                FxPair o;
                kind = fx_pair(dx, pi.rad + pj.rad, (u64)(pi.inv_d + pj.inv_d), ph.fx, o);
                if (kind == FX_LUB && ph.lubrication) {
                    double al = o.alpha, be = o.beta;
                    if (ph.lub_limiter) {
                        // a coefficient near its cap m_ij capfac: compare in FP64
                        const float imf = pi.imf + pj.imf;
                        if (!(fx_approx(be) * imf < capf && fx_approx(al) * imf < capf)) {
                            const double lim = ph.capfac * fx_recip(pi.im + pj.im, imf);
                            if (be > lim) { be = lim; ++nlim; }
                            if (al > lim) { al = lim; ++nlim; }
                        }
                    }
                    double du[3];
#pragma unroll
                    for (int a = 0; a < 3; ++a) du[a] = ri.u[a] - rj.u[a];
                    const double un = du[0] * o.n[0] + du[1] * o.n[1] + du[2] * o.n[2];
                    const double sn = (al - be) * un;
                    const PairRes r = {{sn * o.n[0] - al * du[0], sn * o.n[1] - al * du[1], sn * o.n[2] - al * du[2]}, 1};
                    Bx.pres[sl] = r;
                } else if (kind != FX_EXACT) {
                    Bx.pres[sl].flag = 0;
                }
            }
            if (kind == FX_EXACT) {
                const int q = atomicAdd(&Qs.en, 1);
                if (q < EXACT_CAP) {
                    Qs.eslot[q] = sl;
                    Qs.ei[q] = i;
                    Qs.ej[q] = j;
                } else {
                    exact(sl, i, j);
                }
            }
        };

        int head = 0, qn = 0;  // the warp's ring: qn entries from head
        // outer pairs only once a particle of the box has moved shell/2
        const int parts = Bx.moved[src_tmp] ? 2 : 1;
        // cleared for this substep's update to set, by one thread of the box: a
        // store from every block to the word all blocks read costs 20 us a launch
        if (tl.begin == 0 && threadIdx.x == 0) Bx.moved[1 - src_tmp] = 0;
        for (long long c0 = tl.begin + 32 * wid; c0 < tl.end; c0 += 32 * nw)
        for (int w = 0; w < parts; ++w) {
            const long long p = c0 + lane;
            const bool own = p < tl.end;
            const int h0 = __shfl_sync(0xffffffffu, own ? (w ? Bx.hoff2[p] : Bx.hoff[p]) : 0, 0);
            const int total = __reduce_add_sync(0xffffffffu, own ? (w ? Bx.hn2[p] : Bx.hn[p]) : 0);
            for (int t0 = 0; t0 < total; t0 += 32) {
                const int sl = h0 + t0 + lane;
                bool pass = false;
                int i = 0, j = 0;
                if (t0 + lane < total) {
                    j = Bx.hj[sl];
                    i = (int)c0 + Bx.hl[sl];
                    const float4 pi = fin[i], pj = fin[j];
                    const float fx_ = min_image_f(pj.x - pi.x, Lf[0], g.per[0]);
                    const float fy = min_image_f(pj.y - pi.y, Lf[1], g.per[1]);
                    const float fz = min_image_f(pj.z - pi.z, Lf[2], g.per[2]);
                    const float fr = 0.5f * (pi.w + pj.w) + rng_extra_f + SCREEN_MARGIN;
                    pass = fx_ * fx_ + fy * fy + fz * fz < fr * fr;
                    if (!pass) Bx.pres[sl].flag = 0;
                }
                const unsigned m = __ballot_sync(0xffffffffu, pass);
                if (pass) {
                    const int k = (head + qn + __popc(m & ((1u << lane) - 1))) & 63;
                    Qs.slot[wid][k] = sl;
                    Qs.i[wid][k] = i;
                    Qs.j[wid][k] = j;
                }
                qn += __popc(m);
                __syncwarp();
                if (qn >= 32) {
                    eval(head + lane);
                    head += 32;
                    qn -= 32;
                    __syncwarp();
                }
            }
        }
        if (lane < qn) eval(head + lane);
        __syncthreads();
        const int ne = min(Qs.en, EXACT_CAP);
        for (int q = threadIdx.x; q < ne; q += blockDim.x) exact(Qs.eslot[q], Qs.ei[q], Qs.ej[q]);
        __syncthreads();
        if (threadIdx.x == 0) Qs.en = 0;
        __syncthreads();
        // each capped coefficient acts on both partners (the count of the
        // per-particle evaluation of Sec. 3.1.3)
        if (nlim) atomicAdd(&Bx.counters[CNT_LUB_LIMITED], 2ull * nlim);
    }
}

__global__ void __launch_bounds__(32 * PAIR_WARPS, DPS_PAIRS_MINB)
    k_dem_pairs64(const BoxDev *__restrict__ boxes, const Tile *__restrict__ tiles, int ntiles, int src_tmp) {
    __shared__ PairQueue Qs;
    if (threadIdx.x == 0) Qs.en = 0;
    __syncthreads();
    DPS_FOR_TILES(tiles, ntiles, t) {
        const Tile tl = tiles[t];
        pairs64_tile(boxes[tl.box], tl, src_tmp, Qs);
    }
}

// The sums of a substep and the update: one thread per particle adds the
// forces of its owned pairs (ascending partner), minus those of the pairs its
// lower partners own (ascending owner), each pair's n x F_t times d_i/2, then
// the walls and Eq. particle_motion.  The order depends on the list alone.
// WALLS: some box of the batch has a wall axis (else the wall code is left
// out: 72 registers instead of 168, more warps for a kernel that waits on
// the scattered loads of the pair results)
// A pair's force and flag share one 32-byte record, so an entry costs one
// sector and one dependent load.  (A force plane and a flag array took three
// sectors and two loads.)
#ifndef DPS_GATHER_GC
#define DPS_GATHER_GC 3  // entries whose loads are issued before any is added (4: 1% slower, 6: 4%)
#endif
#ifndef DPS_GATHER_MINB
#define DPS_GATHER_MINB 7  // 128-thread blocks per SM the register budget is sized for
#endif
// slots of a particle's pairs in contact with friction: listed while the forces
// are summed, so that a warp pays for the most contacts of a particle and not
// for every entry at which one of its lanes has one
constexpr int TAN_CAP = 8;
template <bool WALLS>
__device__ __forceinline__ void gather64_tile(const BoxDev &Bx, const Tile &tl, int src_tmp, int key_out,
                                              int (*tan_slot)[128]) {
    {
        const PairRes *pres = Bx.pres;
        const int parts = Bx.moved[src_tmp] ? 2 : 1;
        for (long long i = tl.begin + threadIdx.x; i < tl.end; i += blockDim.x) {
            double F[3] = {0, 0, 0}, T[3] = {0, 0, 0}, T2[3] = {0, 0, 0};
            int nc = 0;  // pairs in contact with friction
            const int *rr = Bx.rrow + i * (long long)Bx.maxn;
            // the entries in chunks of GC: the slot indices and records of a
            // chunk are loaded before any is added; the additions keep the
            // list order
            constexpr int GC = DPS_GATHER_GC;
#pragma unroll 1
            for (int w = 0; w < parts; ++w) {
            const int h0 = w ? Bx.hoff2[i] : Bx.hoff[i], nh = w ? Bx.hn2[i] : Bx.hn[i];
            const int nr = w ? Bx.rn2[i] : Bx.rn[i];
            if (w) rr += Bx.rn[i];
            for (int c0 = 0; c0 < nh + nr; c0 += GC) {
                int sl[GC];
#pragma unroll
                for (int u = 0; u < GC; ++u) {
                    const int c = c0 + u;
                    sl[u] = c < nh ? h0 + c : (c < nh + nr ? rr[c - nh] : -1);
                }
                PairRes r[GC];
#pragma unroll
                for (int u = 0; u < GC; ++u) {
                    r[u].flag = 0;
                    if (sl[u] >= 0) r[u] = pres[sl[u]];
                }
#pragma unroll
                for (int u = 0; u < GC; ++u) {
                    // the owner's force or its opposite on the partner: the sign
                    // is selected, not branched on, since each side of a branch
                    // would issue the three FP64 additions again
                    const u64 sg = c0 + u < nh ? 0ull : 0x8000000000000000ull;
                    if (r[u].flag)
#pragma unroll
                        for (int a = 0; a < 3; ++a) F[a] += fx_double(fx_bits(r[u].F[a]) ^ sg);
                    if (r[u].flag == 2) {  // rare: its n x F_t is added below
                        if (nc < TAN_CAP)
                            tan_slot[nc][threadIdx.x] = sl[u];
                        else
#pragma unroll
                            for (int a = 0; a < 3; ++a) T2[a] += Bx.ptan[3 * (long long)sl[u] + a];
                        ++nc;
                    }
                }
            }
            }
            if (nc) {  // (d_i/2) sum of n x F_t
                for (int q = 0; q < min(nc, TAN_CAP); ++q) {
                    const double *t3 = Bx.ptan + 3 * (long long)tan_slot[q][threadIdx.x];
#pragma unroll
                    for (int a = 0; a < 3; ++a) T[a] += t3[a];
                }
                const double lev = 0.5 * Bx.pf[Bx.cur][PD * Bx.cap + i];
#pragma unroll
                for (int a = 0; a < 3; ++a) T[a] = (T[a] + T2[a]) * lev;
            }
            finish_particle<WALLS, true>(Bx, i, src_tmp, F, T, key_out, Bx.moved + 1 - src_tmp);
        }
    }
}

template <bool WALLS>
__global__ void __launch_bounds__(128, WALLS ? 3 : DPS_GATHER_MINB) k_dem_gather64(const BoxDev *__restrict__ boxes,
                                                        const Tile *__restrict__ tiles, int ntiles, int src_tmp,
                                                        int key_out) {
    __shared__ int tan_slot[TAN_CAP][128];
    DPS_FOR_TILES(tiles, ntiles, t) {
        const Tile tl = tiles[t];
        gather64_tile<WALLS>(boxes[tl.box], tl, src_tmp, key_out, tan_slot);
    }
}

// Boxes of one tile each (up to 128 particles; one sphere settling, a pair
// colliding): a block runs all substeps of its box, a barrier where the general
// path has a launch.  One sphere at 32 x 32 x 64: 8.1 -> 4.9 us a substep.
template <bool WALLS>
__global__ void __launch_bounds__(128) k_dem_solo64(const BoxDev *__restrict__ boxes, const Tile *__restrict__ tiles,
                                                    int n_dem) {
    __shared__ PairQueue Qs;
    __shared__ int tan_slot[TAN_CAP][128];
    const Tile tl = tiles[blockIdx.x];
    const BoxDev &Bx = boxes[tl.box];
    if (threadIdx.x == 0) Qs.en = 0;
    __syncthreads();
#pragma unroll 1
    for (int sd = 0; sd < n_dem; ++sd) {
        pairs64_tile(Bx, tl, sd & 1, Qs);
        __syncthreads();
        gather64_tile<WALLS>(Bx, tl, sd & 1, sd == n_dem - 1, tan_slot);
        __syncthreads();
    }
}

// block: a multiple of 32 and of every tile's lanes (Tile::first).
// rows: 1 also the pair rows of the FP64 form (two more launches), 2 the inner
// rows of the FP16-storage form (one more)
void launch_build_nlist(const BoxDev *boxes, const Tile *tiles, int ntiles, int grid, int block, int rows,
                        cudaStream_t s) {
    k_build_nlist<<<grid, block, 0, s>>>(boxes, tiles, ntiles);
    if (rows == 1) {
        k_half_rows<<<grid, 128, 0, s>>>(boxes, tiles, ntiles);
        k_reverse_slots<<<grid, 128, 0, s>>>(boxes, tiles, ntiles);
    } else if (rows == 2) {
        k_inner_rows<<<grid, 128, 0, s>>>(boxes, tiles, ntiles);
    }
}

// mixed forms; lanes: 1, 2, 4 or 8 lanes per particle, 0: each tile its
// box's (block a multiple of 32); walls: some box has a wall axis
// key_out: the last substep of a subcycle also writes the particles' linked
// cells and their counts for the sort that follows
void launch_dem_substep(const BoxDev *boxes, const Tile *tiles, int ntiles, int src_tmp, int key_out, int lanes,
                        int walls, int grid, int block, cudaStream_t s) {
#define DPS_DEM(L) k_dem_pairsum_mixed<L><<<grid, block, 0, s>>>(boxes, tiles, ntiles, src_tmp)
    if (lanes >= 8) DPS_DEM(8);
    else if (lanes == 4) DPS_DEM(4);
    else if (lanes == 2) DPS_DEM(2);
    else if (lanes == 1) DPS_DEM(1);
    else DPS_DEM(0);
#undef DPS_DEM
    if (walls)
        k_dem_integrate<true><<<grid, 128, 0, s>>>(boxes, tiles, ntiles, src_tmp, key_out);
    else
        k_dem_integrate<false><<<grid, 128, 0, s>>>(boxes, tiles, ntiles, src_tmp, key_out);
}

// FP64 form: the pair kernel, then the gather kernel, over the particle tiles
// of every box (one block per tile: blocks that finish make room for others)
void launch_dem_substep64(const BoxDev *boxes, const Tile *tiles, int ntiles, int src_tmp, int key_out, int walls,
                          int part_tile, cudaStream_t s) {
    const int warps = part_tile < 32 * PAIR_WARPS ? (part_tile + 31) / 32 : PAIR_WARPS;
    k_dem_pairs64<<<ntiles, 32 * warps, 0, s>>>(boxes, tiles, ntiles, src_tmp);
    const int grid = ntiles;
    if (walls)
        k_dem_gather64<true><<<grid, 128, 0, s>>>(boxes, tiles, ntiles, src_tmp, key_out);
    else
        k_dem_gather64<false><<<grid, 128, 0, s>>>(boxes, tiles, ntiles, src_tmp, key_out);
}

// every box is one tile: all substeps in one launch
void launch_dem_solo64(const BoxDev *boxes, const Tile *tiles, int ntiles, int n_dem, int walls, cudaStream_t s) {
    if (walls) k_dem_solo64<true><<<ntiles, 128, 0, s>>>(boxes, tiles, n_dem);
    else k_dem_solo64<false><<<ntiles, 128, 0, s>>>(boxes, tiles, n_dem);
}

// tiles of at most 32 particles with 8 lanes: substeps sd to sd + n - 1 (n > 1:
// every box is one tile)
void launch_dem_mixed8(const BoxDev *boxes, const Tile *tiles, int ntiles, int sd, int n, int n_dem, int walls,
                       cudaStream_t s) {
    if (walls) k_dem_mixed8<true><<<ntiles, 256, 0, s>>>(boxes, tiles, sd, n, n_dem);
    else k_dem_mixed8<false><<<ntiles, 256, 0, s>>>(boxes, tiles, sd, n, n_dem);
}

}  // namespace dps
