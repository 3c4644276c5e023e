// box.cuh -- the device box table.  Every kernel of the coupled step works on
// a list of tiles, each a contiguous range of cells or particles of one box;
// one launch therefore advances any number of boxes of different sizes (the
// single domain is a batch of one box).  Kernels read the box's geometry,
// physics and buffer pointers from the table; per-launch state common to all
// boxes (AA parity, which particle set is current) is passed by value.
#pragma once
#include "dps_internal.cuh"

namespace dps {

// one particle as the FP64 pair kernel reads it (a gather of whole records:
// two 32-byte sectors and one, where the separate planes would take nine)
struct alignas(16) DemRec {
    i64 x[3];      // position in units of 2^-Phys::fx.frac
    double u[3];
};
struct alignas(16) DemPart {
    i64 rad, inv_d;  // fx_radius, fx_inv_d
    double im;       // 1/m
    float imf;
    int pad;
};

// result of a pair and substep: the force on the owner of the slot, and 0: the
// pair did not pass, 1: it did, 2: and its n x F_t is nonzero (BoxDev::ptan)
struct alignas(32) PairRes {
    double F[3];
    i64 flag;
};

struct BoxDev {
    Geom g;
    Phys ph;
    int R;             // neighbour search radius (cells)
    // step state advanced on the device (current particle set, history
    // flags); the AA parity is common to the batch and passed per launch
    int parity, cur, have_uprev, have_usub;
    long long np, cap;
    // fluid
    void *pdf;
    void *eps, *fpf, *fam, *acc, *rho, *j, *uD, *uprev, *gradP, *DuDt;
    void *ire;         // 1/(rho eps_f) of the moments pass (eps_f of the step start)
    void *curl;        // curl of u_f for the lift force: the u_D planes, free after K2b
    // particles: two SoA sets and the DEM ping-pong planes
    double *pf[2];
    int *pi[2];
    double *xtmp;
    float4 *xf[2];     // float (x, y, z, d) of the current set / of the ping-pong planes
    float4 *vf[2];     // float (u, m) likewise
    float4 *of[2];     // float (omega, 0) likewise
    float4 *xs;        // float position at the last sort, and d
    int *nlist;        // Verlet list, row by row (k_build_nlist)
    int *nlist_n, *nlist_o;  // inner and outer partners per particle (one-row form: all, 0)
    int split;         // 1: inner partners from the row's front, outer ones from its back; 0: one row
    int *ilist;        // one-row form: the inner partners, ilist[i*maxi + k], dem_lanes columns, gaps -1
    int *ilist_n;
    int maxi, dem_lanes;
    int *moved;        // [3], by source buffer of a substep (k_dem_mixed8: by substep mod 3): some particle has
                       // moved more than shell/2
    int maxn;          // list capacity per particle
    // FP64 form: the list as unordered pairs, each evaluated once per
    // substep (Newton's third law).  Particle i owns the pairs with its
    // partners j > i: hn[i] of them, in ascending j, at slots hoff[i] ...
    // (hj: the partner of a slot; slots are allocated per block from *ptop).
    // rn[i] / rrow[i*maxn + r]: the slots of the pairs (k, i), k < i, in
    // ascending k.
    int *hj, *hoff, *hn, *rrow, *rn;
    int *hoff2, *hn2, *rn2;  // the same of the outer partners (behind the inner ones in rrow)
    PairRes *pres;
    double *ptan;      // n x F_t of a slot [3] (written where flagged 2)
    unsigned char *hl;  // owner of a slot: its index within the chunk of 32 particles of its tile
    // records of the pair kernel: the dynamic state of the current set / of
    // the ping-pong planes, and the particle constants (set at every sort)
    DemRec *rec[2];
    DemPart *part[2];  // by particle set
    unsigned long long *ptop;
    long long pcap;    // slots
    int ufield;        // 1: the added-mass reaction writes u_f of the subcycle to the u_D planes (FP64 form)
    int lowp;          // 1: low-precision form (FP32 coupling arithmetic)
    float *pwf;        // FP32 kernel weights [9][cap] (low-precision forms)
    float *f32p;       // FP32 copies of F_am (3 planes) and F_d (3 planes) [6][cap]
    double *psum;      // mixed-form DEM: pair sums of a substep, force and torque [6][cap]
    // linked cells
    int *cell_start, *count, *key, *tmp, *perm;
    int *scan_part;    // per scan tile partial sums of this box
    // status
    int *status;
    unsigned long long *counters;
};

struct Tile {
    int box;
    int first;         // index of this tile within its box (scan tiles)
    long long begin, end;
};

// iterate the tiles of a launch: one block per tile, blocks stride over tiles
#define DPS_FOR_TILES(tiles, ntiles, t) for (int t = blockIdx.x; t < (ntiles); t += gridDim.x)

// a brick tile: its origin (any cell of a box of 2^27) and extent (up to 8 an axis)
__host__ __device__ inline Tile brick_tile(int box, int x, int y, int z, int ex, int ey, int ez) {
    return Tile{box, 0, (long long)x | ((long long)y << 32),
                (long long)z | ((long long)ex << 32) | ((long long)ey << 40) | ((long long)ez << 48)};
}
__host__ __device__ __forceinline__ void brick_of(const Tile &t, int &x, int &y, int &z, int &ex, int &ey, int &ez) {
    x = (int)t.begin;
    y = (int)(t.begin >> 32);
    z = (int)t.end;
    ex = (int)(t.end >> 32) & 0xff;
    ey = (int)(t.end >> 40) & 0xff;
    ez = (int)(t.end >> 48) & 0xff;
}

}  // namespace dps
