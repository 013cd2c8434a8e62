// What the relaxation's kernels share: the tile geometry, the shared-memory
// planes that blocks exchange their borders through, the waits for other
// tiles and the requests between them (see k_relax.cu).
#pragma once

#include "epic_internal.cuh"

namespace epic {

namespace {

constexpr int RT_COLS = 64;   // tile width: 16 blocks of four columns
constexpr int RT_BLK = 4;     // a thread's block is 4 x 4 pixels
constexpr int RT_BX = RT_COLS / RT_BLK + 2;   // blocks per plane row, ring included
constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr unsigned long long WAIT_LIMIT_NS = 1000000000ull;  // 1 s

// Threads and plane entries of the instance for tiles of up to MAXR rows.
template <int MAXR>
struct Dim {
    static constexpr int BY = MAXR / RT_BLK, NT = 16 * BY, NB = RT_BX * (BY + 2);
};

// What a solve of a tile did: bit k < 8 = neighbour k (in the order upper
// left, upper, upper right, left, right, lower left, lower, lower right) can
// be improved from the tile's border, TB_ANY = some key of the tile changed.
enum { TB_UL = 1, TB_U = 2, TB_UR = 4, TB_L = 8, TB_R = 16, TB_DL = 32, TB_D = 64, TB_DR = 128, TB_ANY = 256 };

// plane of border cell (r, c) of a block: top row 0-3, bottom row 4-7, left
// column 8-9, right column 10-11
__host__ __device__ constexpr int plane_of(int r, int c) {
    return r == 0 ? c : r == 3 ? 4 + c : c == 0 ? 7 + r : 9 + r;
}

// Entry (r, c) around a thread's block (r or c is -1 or 4) of planes `pl`,
// b = the block's entry.
template <int NB, typename V>
__device__ __forceinline__ V around(const V (*pl)[NB], int b, int r, int c) {
    const int dr = r < 0 ? -1 : r > 3 ? 1 : 0, dc = c < 0 ? -1 : c > 3 ? 1 : 0;
    return pl[plane_of(r & 3, c & 3)][b + dr * RT_BX + dc];
}

// Ring pixel i of a tile with MAXR rows of blocks: 66 above, 66 below, then
// MAXR on either side; its tile coordinates.  Its plane entry is
// plane_of(lr & 3, lc & 3), ring_entry(lr, lc).
template <int MAXR>
constexpr int RING = 2 * (RT_COLS + 2) + 2 * MAXR;
template <int MAXR>
__device__ __forceinline__ void ring_pixel(int i, int *lr, int *lc) {
    if (i < RT_COLS + 2) {
        *lr = -1;
        *lc = i - 1;
    } else if (i < 2 * (RT_COLS + 2)) {
        *lr = MAXR;
        *lc = i - (RT_COLS + 2) - 1;
    } else {
        *lr = (i - 2 * (RT_COLS + 2)) >> 1;
        *lc = (i & 1) ? RT_COLS : -1;
    }
}
__device__ __forceinline__ int ring_entry(int lr, int lc) {
    return ((lr + 4) / 4) * RT_BX + (lc + 4) / 4;
}

// A solve tile: `stack` relaxation tiles of a column (whose seed bins are
// consecutive rows of the tile grid), solved as one.
struct TileGeo {
    int x0, y0;     // image origin
    int wv, rv;     // valid columns (<= 64) and rows
};
__device__ __forceinline__ int solve_rows(const PairDev &P) {   // of solve tiles in a frame
    return P.stack == 2 ? (P.tiles_y + 1) >> 1 : P.tiles_y;
}

__device__ __forceinline__ TileGeo tile_geo(const PairDev &P, int tx, int ty) {
    TileGeo g;
    g.x0 = tx * RT_COLS;
    g.y0 = ty * P.stack * P.tile_h;
    g.wv = min(RT_COLS, P.W - g.x0);
    g.rv = min(P.stack * P.tile_h, P.H - g.y0);
    return g;
}

// A thread's four costs of an image row from offset o on (columns c < ncol;
// zero beyond), with one load where the row allows it.
__device__ __forceinline__ void load_costs(const float *C, size_t o, int ncol, bool vec, float *f) {
    if (ncol >= 4 && vec) {
        const float4 v = __ldg(reinterpret_cast<const float4 *>(C + o));
        f[0] = v.x;
        f[1] = v.y;
        f[2] = v.z;
        f[3] = v.w;
    } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) f[c] = c < ncol ? __ldg(C + o + c) : 0.f;
    }
}
// The same for keys (unreached beyond).  Keys of other tiles may be rewritten
// during the launch: they are read through L2.
__device__ __forceinline__ void load_keys(const pkey_t *K, size_t o, int ncol, bool vec, pkey_t *k) {
    if (ncol >= 4 && vec) {
        const ulonglong2 a = __ldcg(reinterpret_cast<const ulonglong2 *>(K + o));
        const ulonglong2 d = __ldcg(reinterpret_cast<const ulonglong2 *>(K + o + 2));
        k[0] = a.x;
        k[1] = a.y;
        k[2] = d.x;
        k[3] = d.y;
    } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) k[c] = c < ncol ? __ldcg(K + o + c) : KEY_INF;
    }
}

// Where a tile's keys are staged from: the frame's map.
struct FrameMap {
    const pkey_t *keys;
    int W;
    __device__ __forceinline__ explicit FrameMap(const PairDev &P) : keys(P.keys), W(P.W) {}
    // four keys of row y from column x on (columns < ncol)
    __device__ __forceinline__ void row(int x, int y, int ncol, pkey_t *k) const {
        load_keys(keys, (size_t)y * W + x, ncol, (W & 1) == 0, k);
    }
    __device__ __forceinline__ pkey_t at(int x, int y) const { return __ldcg(keys + (size_t)y * W + x); }
};

// The half-cost of a staged cost (half_cost_s with the pair's factors).
struct HalfCost {
    float limit, scale;
    bool bad;
    unsigned largest;
    __device__ __forceinline__ explicit HalfCost(const PairDev &P) {
        const int us = unit_shift(P);
        limit = __int_as_float((128 + us) << 23);   // C_MAX 2^us
        scale = __int_as_float((157 - us) << 23);   // 2^(30 - us)
        bad = false;
        largest = 0;
    }
    __device__ __forceinline__ unsigned operator()(float c) {
        if (!(c >= 0.f && c < limit)) {
            bad = true;
            return 0u;
        }
        const unsigned h = __float2uint_rn(__fmul_rn(c, scale));
        largest = max(largest, h);
        return h;
    }
};

__device__ __forceinline__ unsigned long long wait_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Waits until the four edge neighbours of tile (tx, ty) (those inside the
// tile grid) carry a stamp of this run, i.e. are written; thread k < 4
// watches one.  Gives up after `limit` ns with EPIC_ERR_TIMEOUT (false in every
// thread).
__device__ bool wait_edge_neighbours(const PairDev &P, int tx, int ty, RunState *st,
                                     unsigned long long limit = WAIT_LIMIT_NS) {
    bool gave_up = false;
    const int k = threadIdx.x;
    if (k < 4) {
        const int x = tx + (k == 0 ? -1 : k == 1 ? 1 : 0);
        const int y = ty + (k == 2 ? -1 : k == 3 ? 1 : 0);
        if (x >= 0 && x < P.tiles_x && y >= 0 && y < solve_rows(P)) {
            const unsigned *sp = reinterpret_cast<const unsigned *>(P.tile_stamp + y * P.tiles_x + x);
            const unsigned long long t0 = wait_ns();
            while (ld_acquire(sp) == (unsigned)STAMP_PENDING) {
                if (wait_ns() - t0 > limit) {
                    set_status(st, EPIC_ERR_TIMEOUT);
                    gave_up = true;
                    break;
                }
            }
        }
        __threadfence();
    }
    return __syncthreads_or(gave_up) == 0;
}

// Waits until tile (tx, ty) and its eight neighbours (those inside the tile
// grid) carry a stamp of this run (phase 1 has written them); thread k < 8
// watches neighbour k, thread 8 the tile.  Gives up after `limit` ns with
// EPIC_ERR_TIMEOUT (false in every thread).
__device__ bool wait_tile_and_ring(const PairDev &P, int tx, int ty, RunState *st,
                                   unsigned long long limit = WAIT_LIMIT_NS) {
    bool gave_up = false;
    const int k = threadIdx.x;
    if (k < 9) {
        const int x = k == 8 ? tx : tx + (k < 3 ? k - 1 : k < 5 ? 2 * k - 7 : k - 6);
        const int y = k == 8 ? ty : ty + (k < 3 ? -1 : k < 5 ? 0 : 1);
        if (x >= 0 && x < P.tiles_x && y >= 0 && y < solve_rows(P)) {
            const unsigned *sp = reinterpret_cast<const unsigned *>(P.tile_stamp + y * P.tiles_x + x);
            const unsigned long long t0 = wait_ns();
            while (ld_acquire(sp) == (unsigned)STAMP_PENDING) {
                if (wait_ns() - t0 > limit) {
                    set_status(st, EPIC_ERR_TIMEOUT);
                    gave_up = true;
                    break;
                }
            }
        }
        __threadfence();
    }
    return __syncthreads_or(gave_up) == 0;
}

constexpr unsigned long long IDLE_LIMIT_NS = 2000000000ull;  // 2 s

// Solves tiles until nothing is left to do.  Every CTA owns the tiles
// blockIdx.x, blockIdx.x + nblocks, ... and is the only one to solve them.
// A tile has a count of requests (req): one at the start (the sweep),
// and one from every solve of a neighbour whose border can improve it then (a
// solve holds the tile's ring, so it knows the border pixels next door as they
// were or better: without this test 2.7 of 6.3 solves per tile found nothing
// to do).
// A CTA looks at the counts of its tiles, solves those that are not zero in
// turn, and looks again.  q->open counts all requests that are not
// answered: a solve adds its requests to it before it makes them, and takes
// its own off when they are made, so 0 means that nothing is left anywhere.
// No request waits for an answer: a change goes from one tile to the next in
// a write, a fence, an add and the owner's next look.  (A shared queue of
// tiles cost three more round trips to the L2 per solve, and, serving tiles
// in the order of their requests rather than in turns, 6.7 solves per tile
// where turns and that test take 3.6 on the 64-pair mixed batch, after the
// first.)
//
// solve(P, lt, tx, ty) stages and solves a tile, writes its changed keys and
// returns what it did (TB_*; 0: nothing changed), the same in every thread.
// Returns false if the run has an error or nothing moved for `limit` ns.
struct OwnShared {
    unsigned count[32];   // requests of 32 owned tiles
    unsigned dirty;       // those that have any
    int state;            // -1: done, -2: error
};

template <typename Solve>
__device__ bool own_tiles(const BatchArgs &a, RunState *st, TileWork *q, unsigned *req,
                          OwnShared &S, unsigned nblocks, Solve solve,
                          unsigned long long limit = IDLE_LIMIT_NS) {
    const unsigned Tt = (unsigned)a.total_solve;
    const unsigned mine = (Tt - blockIdx.x + nblocks - 1) / nblocks;   // tiles owned
    // solves of the whole run: a pass is two for each of its tiles (a stack
    // counts once), whichever tiles and CTAs they fall to
    const unsigned long long cap = 2ull * (unsigned long long)a.max_passes * (unsigned)a.total_tiles;
    unsigned long long solved = 0;
    const int tid = threadIdx.x;
    unsigned long long t0 = wait_ns();   // thread 0: when something was last seen to move
    unsigned seen = 0;
    for (unsigned k0 = 0;; k0 = k0 + 32 < mine ? k0 + 32 : 0) {
        if (tid < 32) {
            const unsigned k = k0 + tid;
            unsigned v = 0;
            if (k < mine) v = ld_acquire(req + blockIdx.x + k * nblocks);
            const unsigned dirty = __ballot_sync(FULL, v != 0);
            S.count[tid] = v;
            if (tid == 0) {
                S.dirty = dirty;
                S.state = 0;
                if (dirty == 0) {
                    // (the last group of a round looks for the end)
                    if (k0 + 32 >= mine && ld_acquire(reinterpret_cast<unsigned *>(&q->open)) == 0u)
                        S.state = -1;
                    else if (get_status(st) != 0)
                        S.state = -2;
                    else {
                        const unsigned now = *(volatile unsigned *)&q->solves;
                        if (now > cap) {
                            set_status(st, EPIC_ERR_NOT_CONVERGED);
                            S.state = -2;
                        } else if (now != seen) {
                            seen = now;
                            t0 = wait_ns();
                        } else if (wait_ns() - t0 > limit) {
                            set_status(st, EPIC_ERR_TIMEOUT);
                            S.state = -2;
                        }
                        if (mine <= 32) __nanosleep(64);
                    }
                }
            }
        }
        __syncthreads();
        if (S.state == -1) return true;
        if (S.state == -2) return false;
        unsigned dirty = S.dirty;
        while (dirty) {
            const int i = __ffs(dirty) - 1;
            dirty &= dirty - 1;
            const unsigned t = blockIdx.x + (k0 + i) * nblocks;
            const unsigned n = S.count[i];
            if (tid == 0) atomicSub(req + t, n);   // requests from here on count anew
            const int pi = find_pair(a.solve_base, a.npairs, (int)t);
            const PairDev &P = a.pairs[pi];
            const int lt = (int)t - a.solve_base[pi];
            const int tx = lt % P.tiles_x, ty = lt / P.tiles_x;
            const unsigned f = solve(P, lt, tx, ty);
            if (f) {
                bool ask = false;
                int nt = 0;
                if (tid < 8) {
                    const int x = tx + (tid < 3 ? tid - 1 : tid < 5 ? 2 * tid - 7 : tid - 6);
                    const int y = ty + (tid < 3 ? -1 : tid < 5 ? 0 : 1);
                    ask = ((f >> tid) & 1u) && x >= 0 && x < P.tiles_x && y >= 0 && y < solve_rows(P);
                    nt = a.solve_base[pi] + y * P.tiles_x + x;
                }
                if (tid < 32) {
                    const int asked = __popc(__ballot_sync(FULL, ask));
                    if (tid == 0 && asked) atomicAdd(&q->open, asked);
                }
                __threadfence();   // every thread's keys, and the count, before the requests
                __syncthreads();
                if (ask) atomicAdd(req + nt, 1u);
            }
            // (the requests made are counted already, so the order of the next
            // two does not matter)
            if (tid == 0) {
                atomicSub(&q->open, (int)n);
                atomicAdd(&q->solves, 1u);
            }
            if (++solved > cap) {   // (a CTA that never looks at the run's)
                if (tid == 0) set_status(st, EPIC_ERR_NOT_CONVERGED);
                return false;
            }
        }
        __syncthreads();
    }
}

// Cooperative launch of a tile kernel: every CTA resident, at most one per
// tile unless the launch is captured for replay (`fixed_grid`).
inline cudaError_t launch_cooperative(void (*kernel)(const BatchArgs *), int threads, int tiles,
                                      bool fixed_grid, const BatchArgs *dev, const LaunchCfg &lc,
                                      int *grid_used) {
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    int grid = per_sm * lc.num_sms;
    if (!fixed_grid && grid > tiles) grid = tiles;
    if (grid < 1) grid = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.stream = lc.stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (grid_used) *grid_used = grid;
    return cudaLaunchKernelEx(&cfg, kernel, dev);
}

}  // namespace

}  // namespace epic
