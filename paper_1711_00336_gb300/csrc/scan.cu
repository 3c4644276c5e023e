// scan.cu -- exclusive prefix sum of int32 counts (the cell_start array of the
// linked-cell sort).  Reduce-then-scan over tiles of 8192 values: one pass
// writes tile totals, the totals are scanned (recursively), a second pass
// scans each tile and adds its offset.  Integer sums are exact, so the result
// does not depend on the launch shape.
#include "box.cuh"

namespace dps {

constexpr int SCAN_THREADS = 1024;
constexpr int SCAN_ITEMS = 8;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;

__device__ __forceinline__ int warp_incl_scan(int v) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) >= o) v += t;
    }
    return v;
}

// block-wide exclusive scan of one value per thread; total = block sum
template <int THREADS = SCAN_THREADS>
__device__ __forceinline__ int block_excl_scan(int v, int &total) {
    constexpr int NW = THREADS / 32;
    __shared__ int wsum[NW];
    __shared__ int s_total;
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int inc = warp_incl_scan(v);
    if (lane == 31) wsum[wid] = inc;
    __syncthreads();
    if (wid == 0) {
        int t = lane < NW ? wsum[lane] : 0;
        int ti = warp_incl_scan(t);
        if (lane < NW) wsum[lane] = ti - t;  // exclusive prefix of the warp totals
        if (lane == NW - 1) s_total = ti;
    }
    __syncthreads();
    int res = wsum[wid] + inc - v;
    total = s_total;
    __syncthreads();
    return res;
}

__global__ void __launch_bounds__(SCAN_THREADS) k_tile_sums(const int *__restrict__ in, long long n,
                                                             int *__restrict__ sums) {
    long long base = (long long)blockIdx.x * SCAN_TILE;
    int s = 0;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
        long long i = base + (long long)k * SCAN_THREADS + threadIdx.x;
        if (i < n) s += in[i];
    }
    // block reduction
    __shared__ int red[SCAN_THREADS / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        int t = red[threadIdx.x];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (threadIdx.x == 0) sums[blockIdx.x] = t;
    }
}

// exclusive scan of a tile with each thread owning SCAN_ITEMS consecutive values
__global__ void __launch_bounds__(SCAN_THREADS) k_tile_scan(const int *__restrict__ in, long long n,
                                                             const int *__restrict__ offsets,
                                                             int *__restrict__ out, int write_total) {
    long long base = (long long)blockIdx.x * SCAN_TILE + (long long)threadIdx.x * SCAN_ITEMS;
    int v[SCAN_ITEMS];
    int s = 0;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
        long long i = base + k;
        v[k] = i < n ? in[i] : 0;
        s += v[k];
    }
    int total;
    int ex = block_excl_scan(s, total);
    int off = (offsets ? offsets[blockIdx.x] : 0) + ex;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
        long long i = base + k;
        if (i < n) out[i] = off;
        off += v[k];
    }
    // out[n] = grand total, written by the thread that owns the last value
    if (write_total && base <= n - 1 && n - 1 < base + SCAN_ITEMS) out[n] = off;
}

// number of int32 scratch words the scan of n values needs
long long scan_scratch_words(long long n) {
    long long words = 0;
    while (n > SCAN_TILE) {  // per level: tile sums (t) and their scan (t+1)
        long long t = (n + SCAN_TILE - 1) / SCAN_TILE;
        words += 2 * t + 2;
        n = t;
    }
    return words + 1;
}

// out[0..n] = exclusive prefix of in[0..n), out[n] = total.  in and out may
// not alias.  scratch holds scan_scratch_words(n) ints.
void exclusive_scan(const int *in, long long n, int *out, int *scratch, cudaStream_t s) {
    if (n <= 0) {
        cudaMemsetAsync(out, 0, sizeof(int), s);
        return;
    }
    long long tiles = (n + SCAN_TILE - 1) / SCAN_TILE;
    if (tiles == 1) {
        k_tile_scan<<<1, SCAN_THREADS, 0, s>>>(in, n, nullptr, out, 1);
        return;
    }
    int *sums = scratch;                      // tiles values
    int *sums_scanned = scratch + tiles + 1;  // tiles+1 values, then deeper levels
    k_tile_sums<<<(unsigned)tiles, SCAN_THREADS, 0, s>>>(in, n, sums);
    exclusive_scan(sums, tiles, sums_scanned, sums_scanned + tiles + 1, s);
    k_tile_scan<<<(unsigned)tiles, SCAN_THREADS, 0, s>>>(in, n, sums_scanned, out, 1);
}

// ---- batched scan over the box table ----------------------------------------------
// Scan tiles are BSCAN_TILE cells of one box; Tile::first is the tile's index
// inside its box.  Pass 1 writes each tile's count total; pass 2 sums the
// totals before its tile (up to BSCAN_DIRECT of them: one load a thread for
// most boxes) and scans inside the tile; it writes cell_start and its final
// entry, the particle count.  Boxes with more tiles scan the totals in a launch
// of their own.  Two adjacent 16-byte words a thread, one tile a block: 256^3,
// 179 -> 46 us; 32 x 32 x 64, 21 -> 9 us (tiles of 8192 cells, one word at a
// time, three launches).
constexpr int BSCAN_THREADS = 512, BSCAN_ITEMS = 8;
constexpr int BSCAN_TILE = BSCAN_THREADS * BSCAN_ITEMS;
constexpr int BSCAN_DIRECT = 4096;

// the counts of the thread's BSCAN_ITEMS cells (0 past the tile)
__device__ __forceinline__ void bscan_load(const int *__restrict__ count, long long base, long long end,
                                           int v[BSCAN_ITEMS]) {
    if (base + BSCAN_ITEMS <= end) {
#pragma unroll
        for (int q = 0; q < BSCAN_ITEMS / 4; ++q) {
            const int4 c = *(const int4 *)(count + base + 4 * q);
            v[4 * q] = c.x;
            v[4 * q + 1] = c.y;
            v[4 * q + 2] = c.z;
            v[4 * q + 3] = c.w;
        }
    } else {
#pragma unroll
        for (int k = 0; k < BSCAN_ITEMS; ++k) v[k] = base + k < end ? count[base + k] : 0;
    }
}

__global__ void __launch_bounds__(BSCAN_THREADS) k_bscan_sums(const BoxDev *__restrict__ boxes,
                                                               const Tile *__restrict__ tiles) {
    const Tile tl = tiles[blockIdx.x];
    const BoxDev &B = boxes[tl.box];
    int v[BSCAN_ITEMS], s = 0;
    bscan_load(B.count, tl.begin + (long long)threadIdx.x * BSCAN_ITEMS, tl.end, v);
#pragma unroll
    for (int k = 0; k < BSCAN_ITEMS; ++k) s += v[k];
    __shared__ int red[BSCAN_THREADS / 32];
    s = __reduce_add_sync(0xffffffffu, s);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        s = __reduce_add_sync(0xffffffffu, threadIdx.x < BSCAN_THREADS / 32 ? red[threadIdx.x] : 0);
        if (threadIdx.x == 0) B.scan_part[tl.first] = s;
    }
}

// one block per box: exclusive scan of its tile totals, in place
__global__ void __launch_bounds__(BSCAN_THREADS) k_bscan_parts(const BoxDev *__restrict__ boxes, int nboxes) {
    for (int b = blockIdx.x; b < nboxes; b += gridDim.x) {
        const BoxDev &B = boxes[b];
        const long long nt = (B.g.ncell + BSCAN_TILE - 1) / BSCAN_TILE;
        int carry = 0;
        for (long long base = 0; base < nt; base += BSCAN_THREADS) {
            long long i = base + threadIdx.x;
            int v = i < nt ? B.scan_part[i] : 0;
            int total;
            int ex = block_excl_scan<BSCAN_THREADS>(v, total);
            if (i < nt) B.scan_part[i] = carry + ex;
            carry += total;
        }
    }
}

// direct: scan_part holds the totals, else their exclusive scan
__global__ void __launch_bounds__(BSCAN_THREADS) k_bscan_tiles(const BoxDev *__restrict__ boxes,
                                                                const Tile *__restrict__ tiles, int direct) {
    const Tile tl = tiles[blockIdx.x];
    const BoxDev &B = boxes[tl.box];
    const long long n = B.g.ncell;
    const long long base = tl.begin + (long long)threadIdx.x * BSCAN_ITEMS;
    __shared__ int pre[BSCAN_THREADS / 32];
    int v[BSCAN_ITEMS], s = 0, before = 0;
    bscan_load(B.count, base, tl.end, v);
    if (direct) {
        for (int q = threadIdx.x; q < tl.first; q += BSCAN_THREADS) before += B.scan_part[q];
        before = __reduce_add_sync(0xffffffffu, before);
        if ((threadIdx.x & 31) == 0) pre[threadIdx.x >> 5] = before;
    }
#pragma unroll
    for (int k = 0; k < BSCAN_ITEMS; ++k) s += v[k];
    int total;
    int off = block_excl_scan<BSCAN_THREADS>(s, total);  // (its barriers also order pre)
    if (direct) {
#pragma unroll
        for (int q = 0; q < BSCAN_THREADS / 32; ++q) off += pre[q];
    } else {
        off += B.scan_part[tl.first];
    }
    int o[BSCAN_ITEMS];
#pragma unroll
    for (int k = 0; k < BSCAN_ITEMS; ++k) {
        o[k] = off;
        off += v[k];
    }
    if (base + BSCAN_ITEMS <= tl.end) {
#pragma unroll
        for (int q = 0; q < BSCAN_ITEMS / 4; ++q)
            *(int4 *)(B.cell_start + base + 4 * q) = make_int4(o[4 * q], o[4 * q + 1], o[4 * q + 2], o[4 * q + 3]);
    } else {
#pragma unroll
        for (int k = 0; k < BSCAN_ITEMS; ++k)
            if (base + k < tl.end) B.cell_start[base + k] = o[k];
    }
    // off past the box's last cell is the particle count
    if (base <= n - 1 && n - 1 < base + BSCAN_ITEMS) B.cell_start[n] = off;
}

int bscan_launches(int most_tiles) { return most_tiles <= BSCAN_DIRECT ? 2 : 3; }

// most_tiles: scan tiles of the largest box; returns the launches
int launch_bscan(const BoxDev *boxes, int nboxes, const Tile *scan_tiles, int ntiles, int most_tiles, cudaStream_t s) {
    const int direct = bscan_launches(most_tiles) == 2;
    k_bscan_sums<<<ntiles, BSCAN_THREADS, 0, s>>>(boxes, scan_tiles);
    if (!direct) k_bscan_parts<<<nboxes, BSCAN_THREADS, 0, s>>>(boxes, nboxes);
    k_bscan_tiles<<<ntiles, BSCAN_THREADS, 0, s>>>(boxes, scan_tiles, direct);
    return bscan_launches(most_tiles);
}
int scan_tile_cells() { return BSCAN_TILE; }

}  // namespace dps
