// A-2..A-4: tile intersection, key duplication, 64-bit key sort and tile
// ranges (Sec. 2.1, Step 1-2 and Step 2) on sm_103a.
//
// The key of a (tile, Gaussian) pair is tile_id << 32 | float32 bits of the
// depth, with the Gaussian id as the tie-break (equal depths keep id order).
// It is sorted as an MSD radix sort whose first digit is the whole tile id:
//   k_tile_hist     per-CTA tile counts of each Gaussian's rect, summed in
//                   shared memory and written as one row per CTA (grids of
//   k_col_scan      up to 8192 tiles); a column scan over the CTAs gives
//                   each CTA's offset inside every bucket and the tile
//                   totals.  Larger grids count with one global atomic per
//                   key (k_tile_count).
//   k_tile_scan     one CTA: exclusive scan of the tile counts -> bucket
//                   starts, tile ranges, key count, capacity check
//   k_tile_order    one CTA: heavy-first permutation of the tiles (stable)
//                   (with the per-CTA rows, the column scan's last CTA runs
//                   both: k_col_scan_tail)
//   k_tile_scatter  each pair takes a slot of its tile's bucket and writes
//                   the 64-bit remainder key depth_bits << 32 | id there (a
//                   CTA's slots start at its row offset and are dealt out
//                   with shared-memory atomics: no global atomics)
//   k_tile_sort     bucket sort, heavy first: the remainder keys are unique,
//                   so any correct sort of them gives the same result.
//                   One launch, a distribution sort by depth in shared
//                   memory: a warp a bucket of up to 256 keys, 128 threads
//                   up to 1024, 256 up to 2048, a CTA of 512 above, in slabs
//                   of at most 4096 keys where the bucket is longer.  Buckets
//                   whose depths crowd into one bin are merge sorted instead
//                   (in registers and shared memory; above 65536 keys also in
//                   global memory).  The sort writes tile_id << 32 |
//                   depth_bits and the id.
// The scatter order inside a bucket depends on atomics, the output does not.
// Everything stays on the device: the key count is never read by the host.
#include <algorithm>

#include "gs_internal.cuh"

namespace gs {

#define BIN_THREADS 256
#define TS_THREADS 512
#define TS_KEYS 4096             // keys a CTA sorts in shared memory at a time
#define TS_DIST_KEYS 65536       // longer buckets merge sorted runs in global memory

typedef unsigned long long u64;

template <int DT>
__global__ void __launch_bounds__(BIN_THREADS) k_tile_count(gs_camera cam, float alpha_min, const void* __restrict__ splats,
                                                            int64_t n, uint32_t* __restrict__ count) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const Grid grid = make_grid(cam);
    const Geom G = load_geom<DT>(splats, (uint32_t)k);
    int x0, x1, y0, y1;
    if (tile_rect(grid, G, alpha_min, x0, x1, y0, y1) == 0) return;
    for (int ty = y0; ty < y1; ++ty)
        for (int tx = x0; tx < x1; ++tx) atomicAdd(count + ty * grid.TX + tx, 1u);
}

// Shared-memory aggregated forms of the two passes above, for grids of at
// most AGG_MAX_TILES tiles.  CTA c takes `per_cta` consecutive Gaussians:
//   k_tile_hist      counts its pairs per tile in shared memory and writes
//                    the row hist[c][0..T) (no global atomics);
//   k_col_scan       exclusive prefix of hist[.][t] over the CTAs (in place)
//                    and the tile totals;
//   k_tile_scatter_rows  CTA c starts tile t's slots at start[t] +
//                    hist[c][t] and deals them out with shared-memory atomics.
#define AGG_MAX_TILES 8192
// (A constant, not the device's count: it shapes the workspace, whose size is
// asked for before the device that runs the call may be current.)
#define AGG_ROWS 912         // rows of a large map: one wave of six counting CTAs on 152 SMs

template <int DT>
__global__ void __launch_bounds__(BIN_THREADS) k_tile_hist(gs_camera cam, float alpha_min, const void* __restrict__ splats, int64_t n,
                                                           int64_t per_cta, int ntiles, uint32_t* __restrict__ hist) {
    extern __shared__ uint32_t h[];
    for (int t = threadIdx.x; t < ntiles; t += blockDim.x) h[t] = 0;
    __syncthreads();
    const Grid grid = make_grid(cam);
    const int64_t k0 = (int64_t)blockIdx.x * per_cta, k1 = min(n, k0 + per_cta);
    for (int64_t k = k0 + threadIdx.x; k < k1; k += blockDim.x) {
        const Geom G = load_geom<DT>(splats, (uint32_t)k);
        int x0, x1, y0, y1;
        if (tile_rect(grid, G, alpha_min, x0, x1, y0, y1) == 0) continue;
        for (int ty = y0; ty < y1; ++ty)
            for (int tx = x0; tx < x1; ++tx) atomicAdd(h + ty * grid.TX + tx, 1u);
    }
    __syncthreads();
    uint32_t* row = hist + (size_t)blockIdx.x * ntiles;
    for (int t = threadIdx.x; t < ntiles; t += blockDim.x) row[t] = h[t];
}

// Column scan of the per-CTA rows: CTA b takes CS_TILES tiles; its threads
// split the rows into CS_GROUPS consecutive ranges, sum them, scan the partial
// sums in shared memory and write each row's exclusive prefix in place.
__device__ __forceinline__ void col_scan_body(uint32_t* __restrict__ hist, int nrows, int ntiles,
                                              uint32_t* __restrict__ total, int blk) {
    // CTA: CS_TILES tiles x (1024 / CS_TILES) row groups of consecutive rows
    constexpr int CS_TILES = 8, CS_GROUPS = 1024 / CS_TILES;
    __shared__ uint32_t part[CS_GROUPS][CS_TILES + 1];
    const int tx = threadIdx.x % CS_TILES, ty = threadIdx.x / CS_TILES;
    const int t = blk * CS_TILES + tx;
    const int per = (nrows + CS_GROUPS - 1) / CS_GROUPS;
    const int r0 = min(nrows, ty * per), r1 = min(nrows, r0 + per);
    // rows in groups of 8 loads issued back to back (a dependent sum per
    // load would wait out an L2 round trip per row); the first group stays
    // in registers for the prefix pass (the only group when a thread has at
    // most 8 rows: up to 1024 rows)
    uint32_t sum = 0, v0[8];
    if (t < ntiles)
        for (int r = r0; r < r1; r += 8) {
            uint32_t v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = r + k < r1 ? __ldcg(hist + (size_t)(r + k) * ntiles + t) : 0u;
#pragma unroll
            for (int k = 0; k < 8; ++k) sum += v[k];
            if (r == r0) {
#pragma unroll
                for (int k = 0; k < 8; ++k) v0[k] = v[k];
            }
        }
    part[ty][tx] = sum;
    __syncthreads();
    // warp w < CS_TILES scans column w's CS_GROUPS partial sums (4 per lane)
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (w < CS_TILES) {
        uint32_t v[CS_GROUPS / 32];
        uint32_t loc = 0;
#pragma unroll
        for (int k = 0; k < CS_GROUPS / 32; ++k) {
            v[k] = part[lane * (CS_GROUPS / 32) + k][w];
            loc += v[k];
        }
        uint32_t incl = loc;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        uint32_t run = incl - loc;
#pragma unroll
        for (int k = 0; k < CS_GROUPS / 32; ++k) {
            part[lane * (CS_GROUPS / 32) + k][w] = run;
            run += v[k];
        }
        const int tc = blk * CS_TILES + w;
        if (lane == 31 && tc < ntiles) total[tc] = incl;
    }
    __syncthreads();
    uint32_t run = part[ty][tx];
    if (t < ntiles)
        for (int r = r0; r < r1; r += 8) {
            uint32_t v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k)
                v[k] = r == r0 ? v0[k] : (r + k < r1 ? __ldcg(hist + (size_t)(r + k) * ntiles + t) : 0u);
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (r + k < r1) {
                    hist[(size_t)(r + k) * ntiles + t] = run;
                    run += v[k];
                }
        }
}

__global__ void __launch_bounds__(1024) k_col_scan(uint32_t* __restrict__ hist, int nrows, int ntiles,
                                                   uint32_t* __restrict__ total) {
    col_scan_body(hist, nrows, ntiles, total, (int)blockIdx.x);
}

// Heavy-first tile order (defined below with the tile scan).
template <int NW>
__device__ __forceinline__ void tile_order_body(const uint32_t* __restrict__ ranges, int ntiles,
                                                uint32_t* __restrict__ order, uint32_t* __restrict__ n_big);

template <int DT>
__global__ void __launch_bounds__(BIN_THREADS) k_tile_scatter_rows(gs_camera cam, float alpha_min, const void* __restrict__ splats,
                                                                   int64_t n, int64_t per_cta, int ntiles,
                                                                   const uint32_t* __restrict__ start,
                                                                   const uint32_t* __restrict__ hist, int64_t cap,
                                                                   u64* __restrict__ keys,
                                                                   const uint32_t* __restrict__ ranges,
                                                                   uint32_t* __restrict__ order,
                                                                   uint32_t* __restrict__ n_big) {
    if (blockIdx.x == gridDim.x - 1) {  // the heavy-first order, beside the scatter
        tile_order_body<BIN_THREADS / 32>(ranges, ntiles, order, n_big);
        return;
    }
    extern __shared__ uint32_t h[];
    uint32_t* base = h + ntiles;
    const uint32_t* row = hist + (size_t)blockIdx.x * ntiles;
    for (int t = threadIdx.x; t < ntiles; t += blockDim.x) {
        h[t] = 0;
        base[t] = start[t] + row[t];
    }
    __syncthreads();
    const Grid grid = make_grid(cam);
    const int64_t k0 = (int64_t)blockIdx.x * per_cta, k1 = min(n, k0 + per_cta);
    for (int64_t k = k0 + threadIdx.x; k < k1; k += blockDim.x) {
        const Geom G = load_geom<DT>(splats, (uint32_t)k);
        int x0, x1, y0, y1;
        if (tile_rect(grid, G, alpha_min, x0, x1, y0, y1) == 0) continue;
        const u64 rem = ((u64)__float_as_uint(G.depth) << 32) | (u64)(uint32_t)k;
        for (int ty = y0; ty < y1; ++ty)
            for (int tx = x0; tx < x1; ++tx) {
                const int t = ty * grid.TX + tx;
                const u64 pos = (u64)base[t] + atomicAdd(h + t, 1u);
                if ((int64_t)pos < cap) keys[pos] = rem;
            }
    }
}

// Exclusive scan of the tile counts.  start[t] = min(bucket start, cap);
// ranges (if not NULL) = bucket clipped to the capacity; *n_keys = total.
__device__ __forceinline__ void tile_scan_body(const uint32_t* __restrict__ count, int ntiles, int64_t cap,
                                               uint32_t* __restrict__ start, uint32_t* __restrict__ ranges,
                                               int64_t* __restrict__ n_keys, unsigned int* __restrict__ status) {
    __shared__ u64 s_warp[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    u64 carry = 0;
    // each chunk's counts are loaded while the previous chunk is scanned
    u64 v_nx = (int)threadIdx.x < ntiles ? (u64)__ldcg(count + threadIdx.x) : 0ull;
    for (int base = 0; base < ntiles; base += 1024) {
        const int t = base + threadIdx.x;
        const u64 v = v_nx;
        v_nx = t + 1024 < ntiles ? (u64)__ldcg(count + t + 1024) : 0ull;
        u64 x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const u64 y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_warp[wid] = x;
        __syncthreads();
        if (wid == 0) {
            u64 w = s_warp[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const u64 y = __shfl_up_sync(0xffffffffu, w, o);
                if (lane >= o) w += y;
            }
            s_warp[lane] = w;
        }
        __syncthreads();
        const u64 excl = carry + (wid > 0 ? s_warp[wid - 1] : 0ull) + x - v;
        const u64 total = s_warp[31];
        if (t < ntiles) {
            const u64 b = excl < (u64)cap ? excl : (u64)cap;
            const u64 e = excl + v < (u64)cap ? excl + v : (u64)cap;
            if (start) start[t] = (uint32_t)b;
            if (ranges) {
                ranges[2 * t] = e > b ? (uint32_t)b : 0u;
                ranges[2 * t + 1] = e > b ? (uint32_t)e : 0u;
            }
        }
        carry += total;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        *n_keys = (int64_t)carry;
        if ((int64_t)carry > cap) raise_status(status, GS_ERR_CAPACITY);
    }
}

__global__ void __launch_bounds__(1024) k_tile_scan(const uint32_t* __restrict__ count, int ntiles, int64_t cap,
                                                    uint32_t* __restrict__ start, uint32_t* __restrict__ ranges,
                                                    int64_t* __restrict__ n_keys, unsigned int* __restrict__ status) {
    tile_scan_body(count, ntiles, cap, start, ranges, n_keys, status);
}

// Heavy-first tile order: tiles grouped by quarter octaves of their length
// -- x = length - 1 in [2^m + q 2^(m-2), 2^m + (q + 1) 2^(m-2)), q = 0..3
// (lengths 1 and 0 last) -- longest group first, ascending tile index inside
// a group: a stable counting sort, so the order is a function of the lists
// alone (the compositing kernels may treat the first tiles of the order
// differently, and their results must not depend on scheduling).  Finer than
// whole octaves, it launches the compositing CTAs closer to longest first
// (tracking step 231.6 -> 226.4 us against octaves).  n_big[0..3] receive
// the numbers of tiles longer than 4096, 2048, 1024 and 256 keys, which are
// exactly the first ones of the order (those lengths end groups).
#define OG_N 133  // order groups: quarter octaves of the length, then length 1, then empty
__device__ __forceinline__ int order_group(uint32_t len) {
    if (len == 0) return OG_N - 1;
    const uint32_t x = len - 1u;
    if (x == 0) return OG_N - 2;
    const int msb = 31 - __clz(x);
    const int sub = msb >= 2 ? (int)((x >> (msb - 2)) & 3u) : (int)((x << (2 - msb)) & 3u);
    return (31 - msb) * 4 + (3 - sub);
}

template <int NW>  // warps of the CTA
__device__ __forceinline__ void tile_order_body(const uint32_t* __restrict__ ranges, int ntiles,
                                                uint32_t* __restrict__ order, uint32_t* __restrict__ n_big) {
    __shared__ uint32_t cnt[OG_N], cur[OG_N];
    __shared__ uint32_t wcnt[NW][OG_N];  // per warp and group, within a chunk of 32 NW tiles
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int b = threadIdx.x; b < OG_N; b += blockDim.x) cnt[b] = 0;
    __syncthreads();
    for (int t = threadIdx.x; t < ntiles; t += blockDim.x)
        atomicAdd(&cnt[order_group(__ldcg(ranges + 2 * t + 1) - __ldcg(ranges + 2 * t))], 1u);
    __syncthreads();
    if (warp == 0) {  // exclusive scan of the groups, OG_L a lane
        constexpr int OG_L = (OG_N + 31) / 32;
        uint32_t c[OG_L], sum = 0;
#pragma unroll
        for (int k = 0; k < OG_L; ++k) {
            c[k] = OG_L * lane + k < OG_N ? cnt[OG_L * lane + k] : 0u;
            sum += c[k];
        }
        uint32_t run = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, run, o);
            if (lane >= o) run += y;
        }
        run -= sum;
#pragma unroll
        for (int k = 0; k < OG_L; ++k) {
            const int b = OG_L * lane + k;
            if (b < OG_N) cur[b] = run;
            run += c[k];
            if (b == order_group(4097)) n_big[0] = run;
            if (b == order_group(2049)) n_big[1] = run;
            if (b == order_group(1025)) n_big[2] = run;
            if (b == order_group(257)) n_big[3] = run;
        }
    }
    for (int base = 0; base < ntiles; base += 32 * NW) {
        for (int q = threadIdx.x; q < NW * OG_N; q += blockDim.x) (&wcnt[0][0])[q] = 0;
        __syncthreads();
        const int t = base + (int)threadIdx.x;
        const int grp = t < ntiles ? order_group(__ldcg(ranges + 2 * t + 1) - __ldcg(ranges + 2 * t)) : OG_N;
        const unsigned same = __match_any_sync(0xffffffffu, grp);
        const unsigned rank = __popc(same & ((1u << lane) - 1u));
        if (grp < OG_N && rank == 0) wcnt[warp][grp] = __popc(same);
        __syncthreads();
        for (int b = threadIdx.x; b < OG_N; b += blockDim.x) {  // exclusive scan over the warps, per group
            uint32_t run = cur[b];
            for (int w = 0; w < NW; ++w) {
                const uint32_t v = wcnt[w][b];
                wcnt[w][b] = run;
                run += v;
            }
            cur[b] = run;
        }
        __syncthreads();
        if (grp < OG_N) order[wcnt[warp][grp] + rank] = (uint32_t)t;
        __syncthreads();
    }
}

__global__ void __launch_bounds__(1024) k_tile_order(const uint32_t* __restrict__ ranges, int ntiles,
                                                     uint32_t* __restrict__ order, uint32_t* __restrict__ n_big) {
    tile_order_body<32>(ranges, ntiles, order, n_big);
}

// The column scan followed, in the CTA that finishes last (ticket; every
// other CTA's totals are published before its ticket), by the tile scan and
// the heavy-first order: one launch instead of three.
struct ScanTail {
    unsigned int* ticket;  // zero on entry, zero again on exit
    int64_t cap;
    uint32_t* start;
    uint32_t* ranges;
    int64_t* n_keys;
    unsigned int* status;
    uint32_t* order;
    uint32_t* n_big;
};

__device__ __forceinline__ void col_scan_tail_body(uint32_t* __restrict__ hist, int nrows, int ntiles,
                                                   uint32_t* __restrict__ total, const ScanTail& T, int blk,
                                                   int nblk) {
    __shared__ bool s_last;
    col_scan_body(hist, nrows, ntiles, total, blk);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(T.ticket, 1u) == (unsigned)nblk - 1u;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    tile_scan_body(total, ntiles, T.cap, T.start, T.ranges, T.n_keys, T.status);
    __syncthreads();
    if (T.order) tile_order_body<32>(T.ranges, ntiles, T.order, T.n_big);  // else the scatter's extra CTA
    if (threadIdx.x == 0) *T.ticket = 0u;
}

__global__ void __launch_bounds__(1024) k_col_scan_tail(uint32_t* __restrict__ hist, int nrows, int ntiles,
                                                        uint32_t* __restrict__ total, ScanTail T) {
    col_scan_tail_body(hist, nrows, ntiles, total, T, (int)blockIdx.x, (int)gridDim.x);
}

// k_tile_scatter_rows with the rects the fused projection kept (no
// geometry re-read, no tile-rect arithmetic): only the depth is loaded.
// Block 0 computes the heavy-first order beside the scatter.  The others take
// groups of per_cta Gaussians through the bands of tile rows, one band after
// the other: the keys' 8-byte writes land all over their band's buckets, so a
// band is what L2 holds at once (written as one region of 188 MB, the 23.4 M
// keys of 1920x1080 / 3M took 582 us, 340 MB of it reads of partly written
// lines).
struct ScatterArgs {
    int TX;
    const void* splats;
    int64_t n, per_cta;
    int nrow, ntiles;      // groups of Gaussians; tiles
    int max_rows, stride;  // most tile rows of a band (the shared memory); a block's next band is `stride` on
    const uint32_t* start;
    const uint32_t* hist;
    const uint2* rects;
    int64_t cap;
    u64* keys;
    const int64_t* n_keys;
    const uint32_t* ranges;
    uint32_t* order;
    uint32_t* n_big;
};

// Tile rows per band: one band for every SCATTER_BAND bytes of keys there
// are, at most 6 (every band reads the rects again), and no more rows than
// the shared memory holds.  Scatter times by number of bands: 1200x680 / 1M
// (34 MB of keys) 1 band 55 us, 2 43.7, 4 47, 7 60; 1296x968 / 750k (32 MB) 49,
// 2 40, 3 37, 6 44; 1200x680 / 458k at stride 2 (15 MB) 21.7, 2 19.6; 1920x1080 /
// 3M (188 MB) 3 bands 307, 6 263, 12 277, 24 392.
// From the count on the device, not from the capacity: with room for 16 M
// keys, 1M Gaussians took 32 us at 320x240 (1.5 M keys; 6 bands) and 39 at
// 640x480 (2.5 M); with the count's bands 16 and 24.
#define SCATTER_BAND (13 << 20)
#define SCATTER_SMEM_TILES 6144  // 24 KB

__host__ __device__ inline int scatter_bands(int64_t keys, int TY) {
    const int64_t want = (keys * (int64_t)sizeof(u64) + SCATTER_BAND - 1) / SCATTER_BAND;
    const int most = TY < 6 ? TY : 6;
    return want < 1 ? 1 : want < most ? (int)want : most;
}

template <int DT>
__device__ __forceinline__ void scatter_rects_body(const ScatterArgs& A, int blk) {
    if (blk == 0) {
        tile_order_body<BIN_THREADS / 32>(A.ranges, A.ntiles, A.order, A.n_big);
        return;
    }
    extern __shared__ uint32_t h[];  // next free place of each of the band's tiles
    const int TY = A.ntiles / A.TX, grp = (blk - 1) % A.nrow, band0 = (blk - 1) / A.nrow;
    const int bands = scatter_bands(min(__ldcg(A.n_keys), A.cap), TY), rows = min((TY + bands - 1) / bands, A.max_rows);
    const int64_t k0 = (int64_t)grp * A.per_cta, k1 = min(A.n, k0 + A.per_cta);
    for (int yb = band0 * rows; yb < TY; yb += A.stride * rows) {
        const int t0 = yb * A.TX, nt = min(A.ntiles - t0, rows * A.TX);
        const uint32_t* row = A.hist + (size_t)grp * A.ntiles + t0;
        if (yb != band0 * rows) __syncthreads();  // the last band's places are dealt out
        for (int t = threadIdx.x; t < nt; t += blockDim.x) h[t] = A.start[t0 + t] + row[t];
        __syncthreads();
        for (int64_t kb = k0; kb < k1; kb += blockDim.x) {
            const int64_t k = kb + threadIdx.x;
            int x0 = 0, x1 = 0, y0 = 0, y1 = 0;
            float depth = 0.f;
            if (k < k1) {
                const uint2 r = __ldg(A.rects + k);
                x0 = (int)(r.x & 0xffffu);
                x1 = (int)(r.x >> 16);
                y0 = max((int)(r.y & 0xffffu), yb);
                y1 = max(min((int)(r.y >> 16), yb + rows), y0);
                if (x1 > x0 && y1 > y0)
                    depth = DT == GS_F32 ? __ldg(reinterpret_cast<const float*>(A.splats) + 12 * (size_t)k + 6)
                                         : __ldg(reinterpret_cast<const float*>(A.splats) + 8 * (size_t)k + 2);
            }
            const uint32_t kw = (uint32_t)(kb + (threadIdx.x & ~31u));  // the id: lane o's Gaussian is kw + o
            warp_rect_tiles(x0, y0 - yb, x1 - x0, y1 - y0, __float_as_uint(depth),
                            [&](int tx, int ty, uint32_t d, uint32_t o) {
                const u64 pos = (u64)atomicAdd(h + ty * A.TX + tx, 1u);
                if ((int64_t)pos < A.cap) A.keys[pos] = ((u64)d << 32) | (u64)(kw + o);
            });
        }
    }
}

template <int DT>
__global__ void __launch_bounds__(BIN_THREADS) k_tile_scatter_rects(const ScatterArgs A) {
    scatter_rects_body<DT>(A, (int)blockIdx.x);
}

static int scatter_max_rows(const Grid& g) { return std::min(std::max(SCATTER_SMEM_TILES / g.TX, 1), g.TY); }

// Blocks for this many bands side by side: those of four keys a Gaussian (a
// surface map at up to 1200x680), which the blocks go through in their order
// (3M Gaussians 280 us, one block a group for all six bands 297); a block
// returns at once where there are fewer bands and goes on to another where
// there are more.
static int scatter_stride(const Grid& g, int64_t n, int64_t cap) { return scatter_bands(std::min(cap, 4 * n), g.TY); }

template <int DT>
__global__ void __launch_bounds__(BIN_THREADS) k_tile_scatter(gs_camera cam, float alpha_min, const void* __restrict__ splats,
                                                              int64_t n, const uint32_t* __restrict__ start,
                                                              uint32_t* __restrict__ fill, int64_t cap,
                                                              u64* __restrict__ keys) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const Grid grid = make_grid(cam);
    const Geom G = load_geom<DT>(splats, (uint32_t)k);
    int x0, x1, y0, y1;
    if (tile_rect(grid, G, alpha_min, x0, x1, y0, y1) == 0) return;
    const u64 rem = ((u64)__float_as_uint(G.depth) << 32) | (u64)(uint32_t)k;
    for (int ty = y0; ty < y1; ++ty)
        for (int tx = x0; tx < x1; ++tx) {
            const int t = ty * grid.TX + tx;
            const u64 pos = (u64)start[t] + atomicAdd(fill + t, 1u);
            if ((int64_t)pos < cap) keys[pos] = rem;
        }
}

// Number of keys in sorted run r[0, len) that are < x (lower bound).
__device__ __forceinline__ int rank_in(const u64* r, int len, u64 x) {
    int lo = 0, hi = len;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (__ldcg(r + mid) < x) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// ---------------------------------------------------------------------------
// Merge sort of a bucket with the keys in registers.  Thread t of the
// sorting group holds positions [t KPT, (t+1) KPT) (blocked layout).  Each
// thread first sorts its KPT keys with a register network; then rounds of
// merges double the sorted run length: each thread finds where its KPT
// outputs start in the pair of runs (merge path: a binary search on the
// diagonal) and merges KPT keys serially.  Runs go through shared memory,
// padded by one key per 16 so that the blocked accesses spread over the
// banks.  Padding keys are ~0 (above every real key: depth bits < 2^31).
// ---------------------------------------------------------------------------
__device__ __forceinline__ int pad16(int x) { return x + (x >> 4); }

template <int KPT>
__device__ __forceinline__ void sort_regs(u64 (&v)[KPT]) {
#pragma unroll
    for (int k = 2; k <= KPT; k <<= 1)
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1)
#pragma unroll
            for (int i = 0; i < KPT; ++i) {
                const int p = i ^ j;
                if (p > i) {
                    const u64 lo = v[i] < v[p] ? v[i] : v[p], hi = v[i] < v[p] ? v[p] : v[i];
                    const bool asc = (i & k) == 0;
                    v[i] = asc ? lo : hi;
                    v[p] = asc ? hi : lo;
                }
            }
}

// Barrier of a sorting group: one warp, or nthreads threads on named
// barrier `id`.
__device__ __forceinline__ void group_bar(int id, int nthreads) {
    if (nthreads == 32) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

// Merge rounds from sorted runs of `run` keys up to one run of nthr * KPT
// keys.  t: the thread's index in the group; buf: the group's buffer
// (pad16 of nthr * KPT keys); bar: the group's barrier.
template <int KPT>
__device__ __forceinline__ void merge_rounds(u64 (&v)[KPT], u64* buf, int t, int nthr, int run, int bar) {
    const int M = nthr * KPT;
    for (; run < M; run <<= 1) {
#pragma unroll
        for (int k = 0; k < KPT; ++k) buf[pad16(t * KPT + k)] = v[k];
        group_bar(bar, nthr);
        const int pair0 = (t * KPT) & ~(2 * run - 1);
        const int diag = t * KPT - pair0;
        const int a0 = pair0, b0 = pair0 + run;
        int lo = max(0, diag - run), hi = min(diag, run);
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (buf[pad16(a0 + mid)] < buf[pad16(b0 + diag - 1 - mid)]) lo = mid + 1;
            else hi = mid;
        }
        int i = lo, j = diag - lo;
        u64 x = i < run ? buf[pad16(a0 + i)] : ~0ull;
        u64 y = j < run ? buf[pad16(b0 + j)] : ~0ull;
#pragma unroll
        for (int k = 0; k < KPT; ++k) {
            const bool ta = x < y;
            v[k] = ta ? x : y;
            if (ta) {
                ++i;
                x = i < run ? buf[pad16(a0 + i)] : ~0ull;
            } else {
                ++j;
                y = j < run ? buf[pad16(b0 + j)] : ~0ull;
            }
        }
        group_bar(bar, nthr);
    }
}

// Loads a bucket of n <= nthr * KPT keys into the blocked layout (coalesced
// through buf), padding with ~0.
template <int KPT>
__device__ __forceinline__ void load_blocked(const u64* key, int n, u64 (&v)[KPT], u64* buf, int t, int nthr, int bar) {
    // all KPT global loads are issued before the first shared store
#pragma unroll
    for (int r = 0; r < KPT; ++r) v[r] = t + r * nthr < n ? __ldcg(key + t + r * nthr) : ~0ull;
#pragma unroll
    for (int r = 0; r < KPT; ++r) buf[pad16(t + r * nthr)] = v[r];
    group_bar(bar, nthr);
#pragma unroll
    for (int k = 0; k < KPT; ++k) v[k] = buf[pad16(t * KPT + k)];
    group_bar(bar, nthr);
}

// Writes the sorted bucket (coalesced through buf): tile_id << 32 |
// depth_bits and the id, or with val NULL the remainder keys as they are.
template <int KPT>
__device__ __forceinline__ void store_sorted(u64* key, uint32_t* val, int n, u64 hi, const u64 (&v)[KPT], u64* buf,
                                             int t, int nthr, int bar) {
#pragma unroll
    for (int k = 0; k < KPT; ++k) buf[pad16(t * KPT + k)] = v[k];
    group_bar(bar, nthr);
    for (int x = t; x < n; x += nthr) {
        const u64 w = buf[pad16(x)];
        key[x] = val ? hi | (w >> 32) : w;
        if (val) val[x] = (uint32_t)w;
    }
}

// Merge sort of n <= nthr * 8 keys from src to (key, val) by a group: each
// warp sorts a run of 256, then the group merges the runs.
__device__ __noinline__ void merge_sort_group(const u64* src, u64* key, uint32_t* val, int n, u64 hi, u64* buf, int t,
                                              int nthr, int bar) {
    u64 v[8];
    load_blocked<8>(src, n, v, buf, t, nthr, bar);
    sort_regs<8>(v);
    merge_rounds<8>(v, buf + pad16((t >> 5) * 256), t & 31, 32, 8, bar);
    if (nthr > 32) {
        group_bar(bar, nthr);
        merge_rounds<8>(v, buf, t, nthr, 256, bar);
    }
    store_sorted<8>(key, val, n, hi, v, buf, t, nthr, bar);
}

// ---------------------------------------------------------------------------
// Distribution sort of a bucket of n <= 8 TPG keys by a group of TPG threads.
// The bucket's depth range is cut into at most 8 TPG equal bins (a shift of
// the depth bits' offset from the smallest: monotone, whatever the bits
// mean); the keys are counted per bin, the counts scanned, the keys placed
// bin by bin in shared memory, and each key's place inside its bin is the
// number of smaller keys there (neighbouring threads hold neighbouring
// places, so they read the same few keys).  Surfaces cluster the depths:
// about 8 keys share a bin on the tracking frame, 15 at 3M / 1920x1080.
// Keys of one depth (a wall parallel to the image) go by the range of their
// ids instead: 3196 and 7223 equal depths a tile 99 -> 28 and 101 -> 33 us.  A
// bin of more than DS_MAX_BIN keys (a far outlier) sends the bucket to the
// merge sort.  About 10 instructions a key and pass instead of
// 25 dependent shared-memory loads a key and merge round (8 to 12 rounds):
// 640x480 / 200k (496 k keys) 34.5 -> 13.2 us, 1200x680 / 1M (4.2 M keys)
// 145 -> 54 us, 1920x1080 / 3M (23.4 M keys) 896 -> 332 us (two CTAs per SM;
// 15.4, 74 and 465 us with one, 14.4, 54 and 357 with three, which spill;
// 1024 threads of 4 keys each: 14.4, 62 and 389).
// src may be key (every key is in registers before the first write).
// buf: 8 TPG keys, bin: 8 TPG counters, red: 2 words a warp of the group.
// ---------------------------------------------------------------------------
#define DS_MAX_BIN 256

template <int TPG>
__device__ __forceinline__ void dist_sort_group(const u64* src, u64* key, uint32_t* val, int n, u64 hi, u64* buf,
                                                uint32_t* bin, uint32_t* red, int t, int bar) {
    constexpr int KPT = 8, M = TPG * KPT, W = TPG / 32;
    constexpr int LOGM = TPG == 32 ? 8 : TPG == 128 ? 10 : TPG == 256 ? 11 : 12;
    static_assert(1 << LOGM == M, "bins per group");
    const int lane = t & 31, w = t >> 5;
    u64 v[KPT];
#pragma unroll
    for (int r = 0; r < KPT; ++r)
        if (t + r * TPG < n) v[r] = __ldcg(src + t + r * TPG);
#pragma unroll
    for (int r = 0; r < KPT / 4; ++r) reinterpret_cast<uint4*>(bin)[t + r * TPG] = make_uint4(0u, 0u, 0u, 0u);
    uint32_t lo, up;
    bool ids = false;  // one depth for all keys: the bins cut the range of their ids
    auto word = [&](u64 k) { return ids ? (uint32_t)k : (uint32_t)(k >> 32); };
    auto range = [&] {
        lo = ~0u;
        up = 0u;
#pragma unroll
        for (int r = 0; r < KPT; ++r)
            if (t + r * TPG < n) {
                lo = min(lo, word(v[r]));
                up = max(up, word(v[r]));
            }
        lo = __reduce_min_sync(0xffffffffu, lo);
        up = __reduce_max_sync(0xffffffffu, up);
        if (W > 1) {
            if (lane == 0) {
                red[w] = lo;
                red[W + w] = up;
            }
            group_bar(bar, TPG);
            lo = __reduce_min_sync(0xffffffffu, lane < W ? red[lane] : ~0u);
            up = __reduce_max_sync(0xffffffffu, lane < W ? red[W + lane] : 0u);
        } else {
            __syncwarp();
        }
    };
    range();
    if (up == lo) {  // (group-uniform)
        ids = true;
        group_bar(bar, TPG);
        range();
    }
    const int sh = max(0, 32 - __clz(up - lo) - LOGM);  // (up - lo) >> sh < M
#pragma unroll
    for (int r = 0; r < KPT; ++r)
        if (t + r * TPG < n) atomicAdd(bin + ((word(v[r]) - lo) >> sh), 1u);
    group_bar(bar, TPG);
    // exclusive scan of the counts, 8 consecutive bins a thread
    uint4 b0 = reinterpret_cast<const uint4*>(bin)[2 * t], b1 = reinterpret_cast<const uint4*>(bin)[2 * t + 1];
    const uint32_t big = max(max(max(b0.x, b0.y), max(b0.z, b0.w)), max(max(b1.x, b1.y), max(b1.z, b1.w)));
    const uint32_t sum = b0.x + b0.y + b0.z + b0.w + b1.x + b1.y + b1.z + b1.w;
    uint32_t inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    uint32_t run = inc - sum, most = __reduce_max_sync(0xffffffffu, big);
    if (W > 1) {
        if (lane == 31) red[w] = inc;  // (every thread has read the range)
        if (lane == 0) red[W + w] = most;
        group_bar(bar, TPG);
        const uint32_t x = lane < W ? red[lane] : 0u;
        run += __reduce_add_sync(0xffffffffu, lane < w ? x : 0u);
        most = __reduce_max_sync(0xffffffffu, lane < W ? red[W + lane] : 0u);
    }
    if (most > DS_MAX_BIN) {  // (group-uniform)
        group_bar(bar, TPG);
        merge_sort_group(src, key, val, n, hi, buf, t, TPG, bar);
        return;
    }
    {
        uint4 e0, e1;
        e0.x = run; e0.y = e0.x + b0.x; e0.z = e0.y + b0.y; e0.w = e0.z + b0.z;
        e1.x = e0.w + b0.w; e1.y = e1.x + b1.x; e1.z = e1.y + b1.y; e1.w = e1.z + b1.z;
        reinterpret_cast<uint4*>(bin)[2 * t] = e0;
        reinterpret_cast<uint4*>(bin)[2 * t + 1] = e1;
    }
    group_bar(bar, TPG);
#pragma unroll
    for (int r = 0; r < KPT; ++r)
        if (t + r * TPG < n) buf[atomicAdd(bin + ((word(v[r]) - lo) >> sh), 1u)] = v[r];
    group_bar(bar, TPG);
    // bin[c] now ends bin c, so bin c starts at bin[c - 1]
    for (int p = t; p < n; p += TPG) {
        const u64 k = buf[p];
        const uint32_t c = (word(k) - lo) >> sh;
        const int q0 = c ? (int)bin[c - 1] : 0, q1 = (int)bin[c];
        int pos = q0;
        for (int q = q0; q < q1; ++q) pos += buf[q] < k ? 1 : 0;
        key[pos] = hi | (k >> 32);
        val[pos] = (uint32_t)k;
    }
}

// Shared memory of a sorting CTA: TS_KEYS keys and TS_KEYS counters (the
// merge sort's padding, one key per 16, lies over the counters).
#define TS_SMEM (TS_KEYS * (int)(sizeof(u64) + sizeof(uint32_t)))

// Class sizes of the order (heavy first): n_big[0..3] tiles are longer than
// 4096, 2048, 1024 and 256 keys.
#define N_CLASS 4

// One launch for all buckets, heavy first: a CTA of 512 threads takes one
// bucket of more than 2048 keys, two of more than 1024, four of more than 256
// (128 threads each) or 16 shorter ones (a warp each).
__device__ __forceinline__ void tile_sort_body(const uint32_t* __restrict__ ranges, const uint32_t* __restrict__ order,
                                               const uint32_t* __restrict__ n_big, int ntiles,
                                               u64* __restrict__ keys, uint32_t* __restrict__ vals,
                                               u64* __restrict__ tmp, int blk) {
    extern __shared__ __align__(16) u64 s[];
    __shared__ uint32_t s_red[2 * TS_THREADS / 32], s_cut[TS_DIST_KEYS / 2048 + 2];
    uint32_t* const bins = reinterpret_cast<uint32_t*>(s + TS_KEYS);
    const int tid = (int)threadIdx.x;
    // the class of this CTA and its first tile in the order
    int lim = 0, first = 0, per = 1;
#pragma unroll
    for (int cl = 0; cl <= N_CLASS; ++cl) {
        const int end = cl < N_CLASS ? (int)n_big[cl] : ntiles;
        per = cl < 2 ? 1 : cl == 2 ? 2 : cl == 3 ? 4 : 16;
        const int blocks = (end - first + per - 1) / per;
        if (blk < blocks) {
            lim = end;
            break;
        }
        blk -= blocks;
        first = end;
    }
    if (lim == 0) return;
    const int TPG = TS_THREADS / per, g = tid / TPG, t = tid % TPG;
    const int idx = first + blk * per + g;
    if (idx >= lim) return;
    const int tile = (int)order[idx];
    const uint32_t b = ranges[2 * tile], e = ranges[2 * tile + 1];
    const int n = (int)(e - b);
    if (n <= 0) return;
    const u64 hi = (u64)(uint32_t)tile << 32;
    u64* key = keys + b;
    uint32_t* val = vals + b;
    // the group's slice of the shared memory: 8 TPG keys, then as many counters
    u64* buf = s + (size_t)g * (TS_KEYS / per * 3 / 2);
    uint32_t* bin = reinterpret_cast<uint32_t*>(buf + TS_KEYS / per);
    uint32_t* red = s_red + g * (2 * TPG / 32);
    if (per == 16) return dist_sort_group<32>(key, key, val, n, hi, buf, bin, red, t, 0);
    if (per == 4) return dist_sort_group<128>(key, key, val, n, hi, buf, bin, red, t, 1 + g);
    if (per == 2) return dist_sort_group<256>(key, key, val, n, hi, buf, bin, red, t, 1 + g);
    if (n <= TS_KEYS) return dist_sort_group<512>(key, key, val, n, hi, buf, bin, red, t, 1);
    // Longer buckets: the keys are first placed bin by bin in tmp (4096 bins
    // over the range of the depths, or the ids of one depth), then slabs of whole bins, each starting in its
    // own 2048 places (so at most 2048 keys and one bin), are sorted alone.
    if (n <= TS_DIST_KEYS) {
        for (int i = tid; i < TS_KEYS; i += TS_THREADS) bins[i] = 0u;
        constexpr int W = TS_THREADS / 32;
        const int lane = tid & 31, w = tid >> 5;
        uint32_t lo, up;
        bool ids = false;  // as in dist_sort_group
        auto word = [&](u64 k) { return ids ? (uint32_t)k : (uint32_t)(k >> 32); };
        for (;;) {
            lo = ~0u;
            up = 0u;
            for (int i = tid; i < n; i += TS_THREADS) {
                const uint32_t d = word(__ldcg(key + i));
                lo = min(lo, d);
                up = max(up, d);
            }
            lo = __reduce_min_sync(0xffffffffu, lo);
            up = __reduce_max_sync(0xffffffffu, up);
            if (lane == 0) {
                s_red[w] = lo;
                s_red[W + w] = up;
            }
            __syncthreads();
            lo = __reduce_min_sync(0xffffffffu, lane < W ? s_red[lane] : ~0u);
            up = __reduce_max_sync(0xffffffffu, lane < W ? s_red[W + lane] : 0u);
            if (up != lo) break;  // (CTA-uniform; ids differ)
            ids = true;
            __syncthreads();
        }
        const int sh = max(0, 32 - __clz(up - lo) - 12);
        for (int i = tid; i < n; i += TS_THREADS)
            atomicAdd(bins + ((word(__ldcg(key + i)) - lo) >> sh), 1u);
        __syncthreads();
        uint32_t c[8], sum = 0u, big = 0u;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            c[k] = bins[8 * tid + k];
            sum += c[k];
            big = max(big, c[k]);
        }
        uint32_t inc = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        uint32_t run = inc - sum, most = __reduce_max_sync(0xffffffffu, big);
        if (lane == 31) s_red[w] = inc;
        if (lane == 0) s_red[W + w] = most;
        __syncthreads();
        run += __reduce_add_sync(0xffffffffu, lane < w ? s_red[lane] : 0u);
        most = __reduce_max_sync(0xffffffffu, lane < W ? s_red[W + lane] : 0u);
        if (most <= 2048u) {  // (CTA-uniform)
            // slab q starts at the first bin that starts at or after place
            // 2048 q: the bin before it crosses that place
            uint32_t at = run;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                bins[8 * tid + k] = at;
                const uint32_t nx = at + c[k];
                // places 2048 q in (at, nx]: at most one (a bin holds at most 2048)
                if ((nx >> 11) != (at >> 11)) s_cut[nx >> 11] = nx;
                at = nx;
            }
            const int slabs = (n + 2047) >> 11;
            __syncthreads();
            if (tid == 0) {
                s_cut[0] = 0u;
                s_cut[slabs] = (uint32_t)n;
            }
            u64* const place = tmp + b;
            for (int i = tid; i < n; i += TS_THREADS) {
                const u64 k = __ldcg(key + i);
                place[atomicAdd(bins + ((word(k) - lo) >> sh), 1u)] = k;
            }
            __threadfence_block();
            __syncthreads();
            for (int q = 0; q < slabs; ++q) {
                const uint32_t p0 = s_cut[q], p1 = s_cut[q + 1];
                if (p1 > p0)
                    dist_sort_group<512>(place + p0, key + p0, val + p0, (int)(p1 - p0), hi, buf, bin, red, t, 1);
                __syncthreads();
            }
            return;
        }
        __syncthreads();
    }
    // the longest buckets, and those with a depth shared by more than 2048
    // keys: sorted runs of TS_KEYS, then merged by rank
    for (int c = 0; c < n; c += TS_KEYS) {
        merge_sort_group(key + c, key + c, nullptr, min(TS_KEYS, n - c), hi, s, tid, TS_THREADS, 1);
        __syncthreads();
    }
    __threadfence_block();
    u64* src = key;
    u64* dst = tmp + b;
    for (int run = TS_KEYS; run < n; run <<= 1) {
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            const int pair = i & ~(2 * run - 1);  // run: a power of two
            const int a0 = pair, a1 = min(pair + run, n), b1 = min(pair + 2 * run, n);
            const u64 x = __ldcg(src + i);
            int out;
            if (i < a1) out = pair + (i - a0) + rank_in(src + a1, b1 - a1, x);
            else out = pair + (i - a1) + rank_in(src + a0, a1 - a0, x);
            dst[out] = x;
        }
        __threadfence_block();
        __syncthreads();
        u64* w = src;
        src = dst;
        dst = w;
    }
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const u64 v = __ldcg(src + i);
        vals[b + i] = (uint32_t)v;
        if (src != key) key[i] = hi | (v >> 32);
    }
    __syncthreads();
    if (src == key)
        for (int i = threadIdx.x; i < n; i += blockDim.x) key[i] = hi | (key[i] >> 32);
}

__global__ void __launch_bounds__(TS_THREADS, 2) k_tile_sort(const uint32_t* __restrict__ ranges,
                                                          const uint32_t* __restrict__ order,
                                                          const uint32_t* __restrict__ n_big, int ntiles,
                                                          u64* __restrict__ keys, uint32_t* __restrict__ vals,
                                                          u64* __restrict__ tmp) {
    tile_sort_body(ranges, order, n_big, ntiles, keys, vals, tmp, (int)blockIdx.x);
}

// ---------------------------------------------------------------------------
// Multi-session waves: column scan (+ tile scan and order), scatter and sort
// over every job of a wave (gs_track_wave)
// ---------------------------------------------------------------------------
struct WaveScanJob {
    uint32_t* hist;
    int nrows, ntiles;
    uint32_t* total;
    ScanTail tail;
};

__global__ void __launch_bounds__(1024) k_wave_col_scan_tail(const __grid_constant__ Wave<WaveScanJob> W) {
    const int j = wave_find(W.start, W.n, (int)blockIdx.x);
    const WaveScanJob& J = W.job[j];
    col_scan_tail_body(J.hist, J.nrows, J.ntiles, J.total, J.tail, (int)blockIdx.x - W.start[j],
                       W.start[j + 1] - W.start[j]);
}

__global__ void __launch_bounds__(BIN_THREADS) k_wave_scatter_rects(const __grid_constant__ Wave<ScatterArgs> W) {
    const int j = wave_find(W.start, W.n, (int)blockIdx.x);
    scatter_rects_body<GS_F32>(W.job[j], (int)blockIdx.x - W.start[j]);
}

struct WaveSortJob {
    const uint32_t* ranges;
    const uint32_t* order;
    const uint32_t* n_big;
    int ntiles;
    u64* keys;
    uint32_t* vals;
    u64* tmp;
};

__global__ void __launch_bounds__(TS_THREADS, 2) k_wave_tile_sort(const __grid_constant__ Wave<WaveSortJob> W) {
    const int j = wave_find(W.start, W.n, (int)blockIdx.x);
    const WaveSortJob& J = W.job[j];
    tile_sort_body(J.ranges, J.order, J.n_big, J.ntiles, J.keys, J.vals, J.tmp, (int)blockIdx.x - W.start[j]);
}

// ---------------------------------------------------------------------------
// Workspace layout
// ---------------------------------------------------------------------------
struct BinLayout {
    size_t off_count, off_fill, off_ticket, off_start, off_order, off_nbig, off_hist, off_tmp, zero_bytes, total;
};

static size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// Gaussians per CTA of the aggregated passes: two per thread (half the
// rows of one per thread for the column scan, and 782 -> 391 CTAs fit one
// wave: projection + binning + sort 63.6-64.6 -> 61.6-62.5 us on the
// tracking frame; four per thread 72.8-74.8).  On larger maps as many as make
// the rows one wave (AGG_ROWS; figures at k_project_hist): rows beyond it cost
// the column scan a pass each (3M Gaussians / 8160 tiles, 1824 rows 41.6 us, 912
// 26.5).  More when the rows would pass 2^24 entries (64 MB).
static int64_t agg_per_cta(int64_t n, int ntiles) {
    const int64_t lim = (int64_t)1 << 24;
    int64_t want = (n * (int64_t)ntiles + lim - 1) / lim;
    const int64_t wave = (n + AGG_ROWS - 1) / AGG_ROWS;
    if (want < wave) want = wave;
    return want > 2 * BIN_THREADS ? want : 2 * BIN_THREADS;
}

static BinLayout bin_layout(int64_t n, int64_t cap, int ntiles) {
    BinLayout L;
    size_t o = 0;
    const int64_t per = agg_per_cta(n, ntiles);
    const int64_t rows = n > 0 ? (n + per - 1) / per : 1;
    L.off_count = o; o = align256(o + sizeof(uint32_t) * (size_t)ntiles);
    L.off_fill = o; o = align256(o + sizeof(uint32_t) * (size_t)ntiles);
    L.off_ticket = o; o = align256(o + sizeof(unsigned int));
    L.zero_bytes = o;
    L.off_start = o; o = align256(o + sizeof(uint32_t) * (size_t)ntiles);
    L.off_order = o; o = align256(o + sizeof(uint32_t) * (size_t)ntiles);
    L.off_nbig = o; o = align256(o + N_CLASS * sizeof(uint32_t));
    L.off_hist = o;
    if (ntiles <= AGG_MAX_TILES) o = align256(o + sizeof(uint32_t) * (size_t)ntiles * (size_t)rows);
    L.off_tmp = o; o = align256(o + sizeof(u64) * (size_t)(cap > 0 ? cap : 1));
    L.total = o;
    return L;
}

}  // namespace gs

using namespace gs;

static gs_status bin_common_checks(const gs_config* cfg, const gs_camera* cam, int rec_dtype, const void* splats,
                                   int64_t n, bool size_query) {
    if (!cfg) return set_error(GS_ERR_INVALID_ARG, "config is NULL");
    if (!cam) return set_error(GS_ERR_INVALID_ARG, "camera is NULL");
    if (cam->width <= 0 || cam->height <= 0 || cam->sx < 1 || cam->sy < 1 || cam->width > (1 << 20) ||
        cam->height > (1 << 20))
        return set_error(GS_ERR_INVALID_ARG, "bad camera size or stride");
    if (rec_dtype != GS_F32 && rec_dtype != GS_BF16 && rec_dtype != GS_F16)
        return set_error(GS_ERR_INVALID_ARG, "bad record dtype %d", rec_dtype);
    if (n < 0 || n > (int64_t)0xFFFFFFF0LL) return set_error(GS_ERR_INVALID_ARG, "bad Gaussian count");
    if (!size_query && n > 0 && (!splats || ((uintptr_t)splats & 15)))
        return set_error(GS_ERR_INVALID_ARG, "splats NULL or not 16-byte aligned");
    const Grid g = make_grid(*cam);
    if ((int64_t)g.TX * g.TY > (1 << 26)) return set_error(GS_ERR_INVALID_ARG, "too many tiles");
    return GS_OK;
}

static gs_status set_agg_smem_attrs() {
    static bool done[64] = {false};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && done[dev]) return GS_OK;
    const int bytes = (int)(2 * AGG_MAX_TILES * sizeof(uint32_t));
    bool ok = cudaFuncSetAttribute(k_tile_scatter_rows<GS_F32>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess &&
              cudaFuncSetAttribute(k_tile_scatter_rows<GS_BF16>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess &&
              cudaFuncSetAttribute(k_tile_scatter_rows<GS_F16>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess &&
              cudaFuncSetAttribute(k_tile_scatter_rects<GS_F32>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes / 2) == cudaSuccess &&
              cudaFuncSetAttribute(k_tile_scatter_rects<GS_BF16>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes / 2) == cudaSuccess &&
              cudaFuncSetAttribute(k_tile_scatter_rects<GS_F16>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes / 2) == cudaSuccess &&
              cudaFuncSetAttribute(k_wave_scatter_rects, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes / 2) == cudaSuccess;
    if (!ok) return set_error(GS_ERR_CUDA, "cudaFuncSetAttribute(k_tile_scatter_rows)");
    if (dev >= 0 && dev < 64) done[dev] = true;
    return GS_OK;
}

// Most CTAs of the bucket sort that lists of up to cap keys in all can fill
// (tile_sort_body's classes: one, two, four or 16 tiles a CTA).  A CTA a tile left
// a grid of 47 k tiles and 28 k keys with 44 k CTAs that only look for their
// class (88 us, now 17).
static int64_t sort_blocks(int ntiles, int64_t cap) {
    const int64_t most = cap / 2049 + (cap / 1025 + 1) / 2 + (cap / 257 + 3) / 4 + (ntiles + 15) / 16;
    return std::min<int64_t>(ntiles, most);
}

// The bucket sort of the scattered keys, heavy tiles first.
static gs_status launch_tile_sort(int ntiles, int64_t cap, const uint32_t* tile_ranges, const uint32_t* order,
                                  const uint32_t* n_big, uint64_t* keys_out, uint32_t* vals_out, u64* tmp,
                                  cudaStream_t st) {
    // once per device (not repeated while a graph is being captured)
    static bool attr_done[64] = {false};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64 || !attr_done[dev]) {
        if (cudaFuncSetAttribute(k_tile_sort, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 TS_SMEM) != cudaSuccess)
            return set_error(GS_ERR_CUDA, "cudaFuncSetAttribute(k_tile_sort)");
        if (dev >= 0 && dev < 64) attr_done[dev] = true;
    }
    k_tile_sort<<<(unsigned)sort_blocks(ntiles, cap), TS_THREADS, TS_SMEM, st>>>(
        tile_ranges, order, n_big, ntiles, (u64*)keys_out, vals_out, tmp);
    return check_launch("k_tile_sort");
}

// Tile counts into `count`: per-CTA rows + column scan (rows kept in `hist`
// for the scatter) when the grid is small enough, else direct atomics.
static gs_status launch_count(const gs_camera* cam, float alpha_min, int rec_dtype, const void* splats, int64_t n,
                              uint32_t* count, uint32_t* hist, cudaStream_t st, const ScanTail* tail = nullptr,
                              bool* fused = nullptr) {
    if (fused) *fused = false;
    if (n == 0) return GS_OK;
    const Grid g = make_grid(*cam);
    const int ntiles = g.TX * g.TY;
    if (ntiles <= AGG_MAX_TILES && hist) {
        const int64_t per = agg_per_cta(n, ntiles);
        const unsigned nb = (unsigned)((n + per - 1) / per);
        const size_t sm = sizeof(uint32_t) * (size_t)ntiles;
        if (rec_dtype == GS_F32) k_tile_hist<GS_F32><<<nb, BIN_THREADS, sm, st>>>(*cam, alpha_min, splats, n, per, ntiles, hist);
        else if (rec_dtype == GS_BF16) k_tile_hist<GS_BF16><<<nb, BIN_THREADS, sm, st>>>(*cam, alpha_min, splats, n, per, ntiles, hist);
        else k_tile_hist<GS_F16><<<nb, BIN_THREADS, sm, st>>>(*cam, alpha_min, splats, n, per, ntiles, hist);
        gs_status s;
        if ((s = check_launch("k_tile_hist")) != GS_OK) return s;
        if (tail) {
            k_col_scan_tail<<<(unsigned)((ntiles + 7) / 8), 1024, 0, st>>>(hist, (int)nb, ntiles, count, *tail);
            if (fused) *fused = true;
            return check_launch("k_col_scan_tail");
        }
        k_col_scan<<<(unsigned)((ntiles + 7) / 8), 1024, 0, st>>>(hist, (int)nb, ntiles, count);
        return check_launch("k_col_scan");
    }
    const unsigned nb = (unsigned)((n + BIN_THREADS - 1) / BIN_THREADS);
    if (rec_dtype == GS_F32) k_tile_count<GS_F32><<<nb, BIN_THREADS, 0, st>>>(*cam, alpha_min, splats, n, count);
    else if (rec_dtype == GS_BF16) k_tile_count<GS_BF16><<<nb, BIN_THREADS, 0, st>>>(*cam, alpha_min, splats, n, count);
    else k_tile_count<GS_F16><<<nb, BIN_THREADS, 0, st>>>(*cam, alpha_min, splats, n, count);
    return check_launch("k_tile_count");
}

extern "C" gs_status gs_bin_count(const gs_config* cfg, const gs_camera* cam, int rec_dtype, const void* splats,
                                  int64_t n,
                                  void* workspace, size_t* workspace_bytes, int64_t* n_keys_out,
                                  gs_stream stream) {
    gs_status s;
    if ((s = bin_common_checks(cfg, cam, rec_dtype, splats, n, workspace == nullptr)) != GS_OK) return s;
    if (!workspace_bytes) return set_error(GS_ERR_INVALID_ARG, "workspace_bytes is NULL");
    const Grid g = make_grid(*cam);
    const int ntiles = g.TX * g.TY;
    const BinLayout L = bin_layout(n, 0, ntiles);
    const size_t need = L.off_tmp;
    if (!workspace) { *workspace_bytes = need; return GS_OK; }
    if (*workspace_bytes < need) return set_error(GS_ERR_WORKSPACE, "workspace %zu < %zu", *workspace_bytes, need);
    if (!n_keys_out) return set_error(GS_ERR_INVALID_ARG, "n_keys_out is NULL");
    cudaStream_t st = (cudaStream_t)stream;
    uint32_t* count = (uint32_t*)((char*)workspace + L.off_count);
    uint32_t* hist = ntiles <= AGG_MAX_TILES ? (uint32_t*)((char*)workspace + L.off_hist) : nullptr;
    if (cudaMemsetAsync(count, 0, sizeof(uint32_t) * (size_t)ntiles, st) != cudaSuccess)
        return set_error(GS_ERR_CUDA, "memset counts");
    if ((s = launch_count(cam, cfg->alpha_min, rec_dtype, splats, n, count, hist, st)) != GS_OK) return s;
    unsigned int* err = status_ptr();
    if (!err) return set_error(GS_ERR_CUDA, "status word address");
    k_tile_scan<<<1, 1024, 0, st>>>(count, ntiles, (int64_t)1 << 62, nullptr, nullptr, n_keys_out, err);
    return check_launch("k_tile_scan");
}

extern "C" gs_status gs_bin_sort(const gs_config* cfg, const gs_camera* cam, int rec_dtype, const void* splats,
                                 int64_t n,
                                 int64_t keys_capacity, void* workspace, size_t* workspace_bytes,
                                 uint64_t* keys_out, uint32_t* vals_out, int64_t* n_keys_out,
                                 uint32_t* tile_ranges, uint32_t* tile_order, gs_stream stream) {
    gs_status s;
    if ((s = bin_common_checks(cfg, cam, rec_dtype, splats, n, workspace == nullptr)) != GS_OK) return s;
    if (!workspace_bytes) return set_error(GS_ERR_INVALID_ARG, "workspace_bytes is NULL");
    if (keys_capacity < 0 || keys_capacity >= ((int64_t)1 << 30))
        return set_error(GS_ERR_INVALID_ARG, "keys_capacity must be in [0, 2^30)");
    const Grid grid = make_grid(*cam);
    const int ntiles = grid.TX * grid.TY;
    const BinLayout L = bin_layout(n, keys_capacity, ntiles);
    if (!workspace) { *workspace_bytes = L.total; return GS_OK; }
    if (*workspace_bytes < L.total) return set_error(GS_ERR_WORKSPACE, "workspace %zu < %zu", *workspace_bytes, L.total);
    if (((uintptr_t)workspace & 255) != 0) return set_error(GS_ERR_INVALID_ARG, "workspace not 256-byte aligned");
    if (!n_keys_out || !tile_ranges || (keys_capacity > 0 && (!keys_out || !vals_out)))
        return set_error(GS_ERR_INVALID_ARG, "an output pointer is NULL");
    cudaStream_t st = (cudaStream_t)stream;
    char* ws = (char*)workspace;
    uint32_t* count = (uint32_t*)(ws + L.off_count);
    uint32_t* fill = (uint32_t*)(ws + L.off_fill);
    uint32_t* start = (uint32_t*)(ws + L.off_start);
    u64* tmp = (u64*)(ws + L.off_tmp);
    uint32_t* hist = ntiles <= AGG_MAX_TILES ? (uint32_t*)(ws + L.off_hist) : nullptr;
    if (cudaMemsetAsync(ws, 0, L.zero_bytes, st) != cudaSuccess) return set_error(GS_ERR_CUDA, "memset bin state");
    unsigned int* err = status_ptr();
    if (!err) return set_error(GS_ERR_CUDA, "status word address");
    // the heavy-first order drives the sort; it is returned when asked for
    uint32_t* order = tile_order ? tile_order : (uint32_t*)(ws + L.off_order);
    uint32_t* n_big = (uint32_t*)(ws + L.off_nbig);
    // with per-CTA rows and keys to scatter, the scatter's extra CTA computes
    // the order; otherwise the column scan's last CTA does
    const bool order_beside = ntiles <= AGG_MAX_TILES && n > 0 && keys_capacity > 0;
    const ScanTail tail = {(unsigned int*)(ws + L.off_ticket), keys_capacity, start, tile_ranges, n_keys_out, err,
                           order_beside ? nullptr : order, n_big};
    bool fused = false;
    if ((s = launch_count(cam, cfg->alpha_min, rec_dtype, splats, n, count, hist, st, &tail, &fused)) != GS_OK) return s;
    if (!fused) {
        k_tile_scan<<<1, 1024, 0, st>>>(count, ntiles, keys_capacity, start, tile_ranges, n_keys_out, err);
        if ((s = check_launch("k_tile_scan")) != GS_OK) return s;
        k_tile_order<<<1, 1024, 0, st>>>(tile_ranges, ntiles, order, n_big);
        if ((s = check_launch("k_tile_order")) != GS_OK) return s;
    }
    if (n == 0 || keys_capacity == 0) return GS_OK;
    const float alpha_min = cfg->alpha_min;
    if (ntiles <= AGG_MAX_TILES) {
        if ((s = set_agg_smem_attrs()) != GS_OK) return s;
        const int64_t per = agg_per_cta(n, ntiles);
        const unsigned nb = (unsigned)((n + per - 1) / per);
        const size_t sm = 2 * sizeof(uint32_t) * (size_t)ntiles;
        if (rec_dtype == GS_F32)
            k_tile_scatter_rows<GS_F32><<<nb + 1, BIN_THREADS, sm, st>>>(*cam, alpha_min, splats, n, per, ntiles, start,
                                                                        hist, keys_capacity, (u64*)keys_out,
                                                                        tile_ranges, order, n_big);
        else if (rec_dtype == GS_BF16)
            k_tile_scatter_rows<GS_BF16><<<nb + 1, BIN_THREADS, sm, st>>>(*cam, alpha_min, splats, n, per, ntiles, start,
                                                                         hist, keys_capacity, (u64*)keys_out,
                                                                         tile_ranges, order, n_big);
        else
            k_tile_scatter_rows<GS_F16><<<nb + 1, BIN_THREADS, sm, st>>>(*cam, alpha_min, splats, n, per, ntiles, start,
                                                                        hist, keys_capacity, (u64*)keys_out,
                                                                        tile_ranges, order, n_big);
        if ((s = check_launch("k_tile_scatter_rows")) != GS_OK) return s;
    } else {
        const unsigned nb = (unsigned)((n + BIN_THREADS - 1) / BIN_THREADS);
        if (rec_dtype == GS_F32)
            k_tile_scatter<GS_F32><<<nb, BIN_THREADS, 0, st>>>(*cam, alpha_min, splats, n, start, fill, keys_capacity, (u64*)keys_out);
        else if (rec_dtype == GS_BF16)
            k_tile_scatter<GS_BF16><<<nb, BIN_THREADS, 0, st>>>(*cam, alpha_min, splats, n, start, fill, keys_capacity, (u64*)keys_out);
        else
            k_tile_scatter<GS_F16><<<nb, BIN_THREADS, 0, st>>>(*cam, alpha_min, splats, n, start, fill, keys_capacity, (u64*)keys_out);
        if ((s = check_launch("k_tile_scatter")) != GS_OK) return s;
    }
    return launch_tile_sort(ntiles, keys_capacity, tile_ranges, order, n_big, keys_out, vals_out, tmp, st);
}

// Projection and binning in one call: gs_project, then gs_bin_sort with
// the first binning pass (per-CTA tile rows) done by the projection kernel
// itself and the scatter reading the rects it kept.  Same outputs as the two
// calls.  Workspace: gs_bin_sort's plus 8 bytes per Gaussian.
extern "C" gs_status gs_project_bin_sort(const gs_config* cfg, const gs_camera* cam, const gs_gaussians* g,
                                         int rec_dtype, void* splats, int64_t keys_capacity, void* workspace,
                                         size_t* workspace_bytes, uint64_t* keys_out, uint32_t* vals_out,
                                         int64_t* n_keys_out, uint32_t* tile_ranges, uint32_t* tile_order,
                                         gs_stream stream) {
    gs_status s;
    if ((s = project_checks(cfg, cam, g, rec_dtype)) != GS_OK) return s;
    const int64_t n = g->n;
    if ((s = bin_common_checks(cfg, cam, rec_dtype, splats, n, workspace == nullptr)) != GS_OK) return s;
    if (!workspace_bytes) return set_error(GS_ERR_INVALID_ARG, "workspace_bytes is NULL");
    if (keys_capacity < 0 || keys_capacity >= ((int64_t)1 << 30))
        return set_error(GS_ERR_INVALID_ARG, "keys_capacity must be in [0, 2^30)");
    const Grid grid = make_grid(*cam);
    const int ntiles = grid.TX * grid.TY;
    const BinLayout L = bin_layout(n, keys_capacity, ntiles);
    const size_t off_rects = L.total, total = align256(L.total + sizeof(uint2) * (size_t)(n > 0 ? n : 1));
    if (!workspace) { *workspace_bytes = total; return GS_OK; }
    if (*workspace_bytes < total) return set_error(GS_ERR_WORKSPACE, "workspace %zu < %zu", *workspace_bytes, total);
    if (((uintptr_t)workspace & 255) != 0) return set_error(GS_ERR_INVALID_ARG, "workspace not 256-byte aligned");
    if (!n_keys_out || !tile_ranges || (keys_capacity > 0 && (!keys_out || !vals_out)))
        return set_error(GS_ERR_INVALID_ARG, "an output pointer is NULL");
    if (ntiles > AGG_MAX_TILES || n == 0) {  // no per-CTA rows: the two calls
        if ((s = gs_project(cfg, cam, g, rec_dtype, splats, stream)) != GS_OK) return s;
        size_t wb = *workspace_bytes;
        return gs_bin_sort(cfg, cam, rec_dtype, splats, n, keys_capacity, workspace, &wb, keys_out, vals_out,
                           n_keys_out, tile_ranges, tile_order, stream);
    }
    cudaStream_t st = (cudaStream_t)stream;
    char* ws = (char*)workspace;
    uint32_t* count = (uint32_t*)(ws + L.off_count);
    uint32_t* start = (uint32_t*)(ws + L.off_start);
    u64* tmp = (u64*)(ws + L.off_tmp);
    uint32_t* hist = (uint32_t*)(ws + L.off_hist);
    void* rects = ws + off_rects;
    if (cudaMemsetAsync(ws, 0, L.zero_bytes, st) != cudaSuccess) return set_error(GS_ERR_CUDA, "memset bin state");
    unsigned int* err = status_ptr();
    if (!err) return set_error(GS_ERR_CUDA, "status word address");
    uint32_t* order = tile_order ? tile_order : (uint32_t*)(ws + L.off_order);
    uint32_t* n_big = (uint32_t*)(ws + L.off_nbig);
    // the order is computed beside the scatter unless there is none
    const ScanTail tail = {(unsigned int*)(ws + L.off_ticket), keys_capacity, start, tile_ranges, n_keys_out, err,
                           keys_capacity == 0 ? order : nullptr, n_big};
    const int64_t per = agg_per_cta(n, ntiles);
    const unsigned nb = (unsigned)((n + per - 1) / per);
    if ((s = launch_project_hist(cfg, cam, g, rec_dtype, splats, per, nb, ntiles, hist, rects, st)) != GS_OK) return s;
    k_col_scan_tail<<<(unsigned)((ntiles + 7) / 8), 1024, 0, st>>>(hist, (int)nb, ntiles, count, tail);
    if ((s = check_launch("k_col_scan_tail")) != GS_OK) return s;
    if (keys_capacity == 0) return GS_OK;
    if ((s = set_agg_smem_attrs()) != GS_OK) return s;
    const int rows = scatter_max_rows(grid), stride = scatter_stride(grid, n, keys_capacity);
    const ScatterArgs A = {grid.TX, splats, n, per, (int)nb, ntiles, rows, stride, start, hist, (const uint2*)rects, keys_capacity,
                           (u64*)keys_out, n_keys_out, tile_ranges, order, n_big};
    const unsigned blocks = 1u + nb * (unsigned)stride;
    const size_t sm = sizeof(uint32_t) * (size_t)grid.TX * (size_t)rows;
    if (rec_dtype == GS_F32) k_tile_scatter_rects<GS_F32><<<blocks, BIN_THREADS, sm, st>>>(A);
    else if (rec_dtype == GS_BF16) k_tile_scatter_rects<GS_BF16><<<blocks, BIN_THREADS, sm, st>>>(A);
    else k_tile_scatter_rects<GS_F16><<<blocks, BIN_THREADS, sm, st>>>(A);
    if ((s = check_launch("k_tile_scatter_rects")) != GS_OK) return s;
    return launch_tile_sort(ntiles, keys_capacity, tile_ranges, order, n_big, keys_out, vals_out, tmp, st);
}

// ---------------------------------------------------------------------------
// Wave launchers (gs_track_wave)
// ---------------------------------------------------------------------------
namespace gs {

// The job's binning state inside its gs_project_bin_sort workspace (the same
// layout as the single-session call), after checking the workspace size.
gs_status wave_bin_layout(const gs_track_job& j, WaveBin* out) {
    const Grid grid = make_grid(j.cam);
    const int ntiles = grid.TX * grid.TY;
    const int64_t n = j.g.n;
    if (ntiles > AGG_MAX_TILES) return set_error(GS_ERR_INVALID_ARG, "more than %d tiles", AGG_MAX_TILES);
    const BinLayout L = bin_layout(n, j.keys_capacity, ntiles);
    const size_t total = align256(L.total + sizeof(uint2) * (size_t)n);
    if (!j.bin_workspace || j.bin_workspace_bytes < total)
        return set_error(GS_ERR_WORKSPACE, "bin workspace %zu < %zu bytes", j.bin_workspace_bytes, total);
    if (((uintptr_t)j.bin_workspace & 255) != 0) return set_error(GS_ERR_INVALID_ARG, "bin workspace not 256-byte aligned");
    char* ws = (char*)j.bin_workspace;
    out->per = agg_per_cta(n, ntiles);
    out->nb = (unsigned)((n + out->per - 1) / out->per);
    out->ntiles = ntiles;
    out->count = (uint32_t*)(ws + L.off_count);
    out->start = (uint32_t*)(ws + L.off_start);
    out->hist = (uint32_t*)(ws + L.off_hist);
    out->ticket = (unsigned int*)(ws + L.off_ticket);
    out->n_big = (uint32_t*)(ws + L.off_nbig);
    out->tmp = ws + L.off_tmp;
    out->rects = ws + L.total;
    return GS_OK;
}

gs_status wave_bin_sort(const gs_track_job* jobs, const WaveBin* bins, int n, cudaStream_t st) {
    unsigned int* err = status_ptr();
    if (!err) return set_error(GS_ERR_CUDA, "status word address");
    gs_status s;
    {
        Wave<WaveScanJob> W;
        W.n = n;
        int blocks = 0;
        for (int j = 0; j < n; ++j) {
            const gs_track_job& t = jobs[j];
            const WaveBin& b = bins[j];
            W.start[j] = blocks;
            blocks += (b.ntiles + 7) / 8;
            const ScanTail tail = {b.ticket, t.keys_capacity, b.start, t.tile_ranges, t.n_keys, err, nullptr, b.n_big};
            W.job[j] = WaveScanJob{b.hist, (int)b.nb, b.ntiles, b.count, tail};
        }
        W.start[n] = blocks;
        k_wave_col_scan_tail<<<(unsigned)blocks, 1024, 0, st>>>(W);
        if ((s = check_launch("k_wave_col_scan_tail")) != GS_OK) return s;
    }
    {
        if ((s = set_agg_smem_attrs()) != GS_OK) return s;
        Wave<ScatterArgs> W;
        W.n = n;
        int blocks = 0, smax = 1;
        for (int j = 0; j < n; ++j) {
            const gs_track_job& t = jobs[j];
            const WaveBin& b = bins[j];
            const Grid g = make_grid(t.cam);
            const int rows = scatter_max_rows(g), stride = scatter_stride(g, t.g.n, t.keys_capacity);
            W.start[j] = blocks;
            blocks += 1 + (int)b.nb * stride;
            smax = std::max(smax, g.TX * rows);
            W.job[j] = ScatterArgs{g.TX, t.splats, t.g.n, b.per, (int)b.nb, b.ntiles, rows, stride, b.start, b.hist,
                                   (const uint2*)b.rects, t.keys_capacity, (u64*)t.keys, t.n_keys, t.tile_ranges,
                                   t.tile_order, b.n_big};
        }
        W.start[n] = blocks;
        k_wave_scatter_rects<<<(unsigned)blocks, BIN_THREADS, sizeof(uint32_t) * (size_t)smax, st>>>(W);
        if ((s = check_launch("k_wave_scatter_rects")) != GS_OK) return s;
    }
    {
        static bool attr_done[64] = {false};
        int dev = 0;
        cudaGetDevice(&dev);
        const int sm = TS_SMEM;
        if (dev < 0 || dev >= 64 || !attr_done[dev]) {
            if (cudaFuncSetAttribute(k_wave_tile_sort, cudaFuncAttributeMaxDynamicSharedMemorySize, sm) != cudaSuccess)
                return set_error(GS_ERR_CUDA, "cudaFuncSetAttribute(k_wave_tile_sort)");
            if (dev >= 0 && dev < 64) attr_done[dev] = true;
        }
        Wave<WaveSortJob> W;
        W.n = n;
        int blocks = 0;
        for (int j = 0; j < n; ++j) {
            const gs_track_job& t = jobs[j];
            const WaveBin& b = bins[j];
            W.start[j] = blocks;
            blocks += (int)sort_blocks(b.ntiles, t.keys_capacity);
            W.job[j] = WaveSortJob{t.tile_ranges, t.tile_order, b.n_big, b.ntiles, (u64*)t.keys, t.vals, (u64*)b.tmp};
        }
        W.start[n] = blocks;
        k_wave_tile_sort<<<(unsigned)blocks, TS_THREADS, (size_t)sm, st>>>(W);
        if ((s = check_launch("k_wave_tile_sort")) != GS_OK) return s;
    }
    return GS_OK;
}

}  // namespace gs
