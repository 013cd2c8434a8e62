// Stage (a) of the interpolator: geodesic assignment map L and distance D
// (Sec. 3.4 "Geodesic Voronoi diagram"; D_G of Eq. 3 on the 8-connected
// grid).  The keys are the same exact fixed-point (D, L) keys as in k_dt.cu,
// so any order of relaxation steps that ends when no step improves any key
// reaches the same keys bit for bit.
//
// One launch holds all of it (a cooperative launch, every CTA resident), in
// five phases:
//   fresh   the distances of every tile from its own seeds (relax_dist.cuh),
//           in two halves of a chessboard: first the tiles with tx + ty even,
//           with unreached neighbours around them, then the others, with the
//           first half's results in their ring (so their solves start from
//           distances that already cross the tile borders, and fewer
//           re-solves follow);
//   spread  every tile is solved again, by the CTA that owns it, whenever a
//           neighbour's border improves it (own_tiles in relax_tiles.cuh),
//           until the distances stand;
//   roots   every reached pixel that is not a seed has a neighbour on a
//           shortest path to it (D(q) + w(q, p) = D(p)).  Following these
//           parents leads to the pixel's seed, or out of the tile; they are
//           followed by pointer jumping in shared memory (a path in a tile is
//           up to ~60 steps long: six jumps).  Pixels rooted in the tile get
//           their label, the others the pixel outside that their path leads
//           to;
//   chains  those are followed (their distances fall, so the chain ends,
//           after a tile or two) to a label.  Nothing else may change a key
//           meanwhile: a pixel that took its label from a chain that another
//           tile improves would not be asked to look again.
//   settle  relaxation of the packed (D, L) keys to the fixed point
//           (relax_settle.cuh).  The keys it starts from are nearly there:
//           every key is the cost and the seed of a real path, so the fixed
//           point, which is unique, is reached from them bit for bit, and
//           where they are final already one round per tile finds nothing to
//           do.  What is left to it: pixels whose shortest paths lead to
//           different matches at the same distance (the smallest index has to
//           win), pixels outside a tile's distance window, and plateaus of
//           cost zero (a pixel whose parent is not strictly nearer is given
//           up by the look for roots).
// Pairs of costs so high that a tile's window holds few steps (settles_only in
// epic_internal.cuh) are settled from their seeds: the other phases would be
// passed through for nothing (eight pairs of constant cost 1.0: relaxation 405
// -> 328 us, the call 880 -> 802).
// Carrying labels through every round of the first two phases instead makes
// each of their steps five times as expensive (see relax_dist.cuh): that form
// took 5.8 ms for the 64-pair mixed batch, this one 4.17 ms.  The form before,
// one warp stepping through the rows of a 64 x 16 tile and closing each along
// itself, ran ~118 dependent row steps per fresh tile and took 4.35 ms for the
// batch; on single frames, where the chain of solves from tile to tile counts,
// it took 199 us on a 256 x 128 pair, 308 us on 1024 x 436, 365 us on 1242 x 375
// and 549 us on 2048 x 1024 against 90, 147, 137 and 214 us now (the stage's
// events in turn).  What bounds it now: latency (12 warps per SM at 168
// registers, 26 % of the issue slots: barriers in the CTA 31 % of the stalls, L2
// loads 14 %, instruction fetch 14 %, dependent integer steps 13 %).  The
// settling sets the registers and spills ~200 bytes of stores and ~300 of loads
// at them; the distances alone need no spill.
//
// Within a phase, and from fresh to spread, nothing waits for the whole grid:
// a second-half tile waits for its four edge neighbours' stamps, and a spread
// solve for the stamps of the tile and its eight neighbours (every wait
// bounded; the prepare kernel marks the tiles pending at the start of a run).
// The spread ends when no request is open, which is also the barrier before
// the roots; grid barriers divide the last three phases.
#include "relax_dist.cuh"
#include "relax_settle.cuh"

namespace epic {

namespace {

constexpr int ROOT_PITCH = RT_COLS + 2;

// A tile with its ring, a cell a pixel.
template <int MAXR>
struct RootCells {
    static constexpr int N = (MAXR + 2) * ROOT_PITCH;
    unsigned lab[N];           // seed labels
    unsigned short par[N];     // parents, then ancestors
};

// The chains of tile (tx, ty)'s pixels that are rooted outside it (about a
// quarter of them: they are listed first, so that every thread has some to
// follow, ChaseList::PER at a time for their loads to overlap).  Pixels of a
// chain may be completed meanwhile: a key is read whole, before or after.
template <int MAXR>
struct ChaseList {
    static constexpr int PER = 4;
    pkey_t key[RT_COLS * MAXR];
    unsigned short at[RT_COLS * MAXR];   // row * 64 + column
    int n;
};

template <int MAXR>
union RelaxShared {
    struct {
        DistTile<MAXR> dist;
        RootCells<MAXR> root;
    };
    ChaseList<MAXR> chase;
    SettleTile<MAXR> settle;
};
static_assert(sizeof(RelaxShared<32>) <= 48 * 1024, "a tile fits in static shared memory");

// The labels of tile (tx, ty)'s seeds, the smallest of those on a pixel.
template <int MAXR>
__device__ __forceinline__ void seed_labels(const PairDev &P, int tx, int ty, const TileGeo &g, RootCells<MAXR> &R) {
    constexpr int NT = Dim<MAXR>::NT;
    for (int q = 0; q < P.stack && ty * P.stack + q < P.tiles_y; ++q) {
        const int bin = (ty * P.stack + q) * P.tiles_x + tx;
        for (int s = P.tile_start[bin] + threadIdx.x, s1 = P.tile_start[bin + 1]; s < s1; s += NT) {
            const int m = P.tile_seeds[s];
            const float4 mt = __ldg(P.matches + m);
            const int px = (int)floorf(mt.x + 0.5f) - g.x0;
            const int py = (int)floorf(mt.y + 0.5f) - g.y0;
            if (px >= 0 && px < g.wv && py >= 0 && py < g.rv)
                atomicMin(&R.lab[(py + 1) * ROOT_PITCH + px + 1], (unsigned)m);
        }
    }
}

// The keys that the settling of tile (tx, ty), local index t, starts from when
// it is all of the relaxation: its seeds', and unreached elsewhere.
template <int MAXR>
__device__ void seed_tile(const PairDev &P, int t, int tx, int ty, RootCells<MAXR> &R, RunState *st) {
    constexpr int NT = Dim<MAXR>::NT;
    const TileGeo g = tile_geo(P, tx, ty);
    for (int i = threadIdx.x; i < RootCells<MAXR>::N; i += NT) R.lab[i] = LABEL_NONE;
    __syncthreads();
    seed_labels(P, tx, ty, g, R);
    __syncthreads();
    for (int i = threadIdx.x; i < RT_COLS * g.rv; i += NT) {
        const int r = i / RT_COLS, c = i % RT_COLS;
        const unsigned m = R.lab[(r + 1) * ROOT_PITCH + c + 1];
        if (c < g.wv) P.keys[(size_t)(g.y0 + r) * P.W + g.x0 + c] = m == LABEL_NONE ? KEY_INF : make_key(0ull, m);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        *(volatile int *)(P.tile_stamp + t) = 0;
        __threadfence();
        atomicAdd(&st->fresh_done, 1u);
    }
}

// The roots of tile (tx, ty)'s pixels.
template <int MAXR>
__device__ void root_tile(const PairDev &P, int tx, int ty, DistTile<MAXR> &T, RootCells<MAXR> &R,
                          RunState *st) {
    constexpr int NT = Dim<MAXR>::NT;
    const int tid = threadIdx.x, bx = tid & 15, by = tid >> 4;
    const int b = (by + 1) * RT_BX + bx + 1;
    const TileGeo g = tile_geo(P, tx, ty);
    const int W = P.W;
    DistBlock B;
    Staged S;
    for (int i = tid; i < RootCells<MAXR>::N; i += NT) {
        R.lab[i] = LABEL_NONE;
        R.par[i] = (unsigned short)i;
    }
    stage_dist(P, tx, ty, g, T, B, S, st, ROOT, FrameMap(P));
    seed_labels(P, tx, ty, g, R);
    block_weights(T, b, S, B);
    __syncthreads();
    const int i0 = (4 * by + 1) * ROOT_PITCH + 4 * bx + 1;   // this block's first cell
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const unsigned dp = B.d[r][c];
            int off = 0;
            // (weights outside the window are capped beyond any difference)
            auto look = [&](int dr, int dc, unsigned w) {
                const int r2 = r + dr, c2 = c + dc;
                const unsigned dq = r2 >= 0 && r2 < 4 && c2 >= 0 && c2 < 4 ? B.d[r2 & 3][c2 & 3]
                                                                         : around(T.d, b, r2, c2);
                if (dp - dq == w && dq < dp) off = dr * ROOT_PITCH + dc;
            };
            look(-1, -1, B.wb[r][c]);
            look(-1, 1, B.ws[r][c + 1]);
            look(1, -1, B.ws[r + 1][c]);
            look(1, 1, B.wb[r + 1][c + 1]);
            look(-1, 0, B.wv[r][c]);
            look(1, 0, B.wv[r + 1][c]);
            look(0, -1, B.wh[r][c]);
            look(0, 1, B.wh[r][c + 1]);
            const int i = i0 + r * ROOT_PITCH + c;
            if (off && dp < S.win && 4 * by + r < g.rv && R.lab[i] == LABEL_NONE)
                R.par[i] = (unsigned short)(i + off);
        }
    __syncthreads();
    // pointer jumping (a jump may read a pointer before or after its own jump:
    // either is an ancestor); 2^12 steps cover any path of a tile
    unsigned anc[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) anc[j] = R.par[i0 + (j >> 2) * ROOT_PITCH + (j & 3)];
    for (int it = 0; it < 12; ++it) {
        unsigned q[16];
        bool moved = false;
#pragma unroll
        for (int j = 0; j < 16; ++j) q[j] = R.par[anc[j]];
#pragma unroll
        for (int j = 0; j < 16; ++j)
            if (q[j] != anc[j]) {
                anc[j] = q[j];
                R.par[i0 + (j >> 2) * ROOT_PITCH + (j & 3)] = (unsigned short)q[j];
                moved = true;
            }
        if (!__syncthreads_or(moved)) break;
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        if (4 * by + r >= g.rv || r >= S.nrow) continue;
        pkey_t *dst = P.keys + (size_t)(g.y0 + 4 * by + r) * W + g.x0 + 4 * bx;
        pkey_t k[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int q = (int)anc[4 * r + c];
            const int qr = q / ROOT_PITCH - 1, qc = q % ROOT_PITCH - 1;
            const bool exits = qr < 0 || qr >= g.rv || qc < 0 || qc >= g.wv;
            const unsigned m = R.lab[q];   // the label of a seed, or none
            const pkey_t d = (S.base + B.d[r][c]) << LABEL_BITS;
            k[c] = exits ? FLAG | d | (unsigned)q : m == LABEL_NONE ? KEY_INF : d | m;
        }
        if (S.ncol >= 4 && (W & 1) == 0) {
            reinterpret_cast<ulonglong2 *>(dst)[0] = make_ulonglong2(k[0], k[1]);
            reinterpret_cast<ulonglong2 *>(dst)[1] = make_ulonglong2(k[2], k[3]);
        } else {
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (c < S.ncol) dst[c] = k[c];
        }
    }
    __syncthreads();
}

template <int MAXR>
__device__ void chase_tile(const PairDev &P, int tx, int ty, ChaseList<MAXR> &Q) {
    constexpr int NT = Dim<MAXR>::NT, PER = ChaseList<MAXR>::PER;
    const int tid = threadIdx.x, bx = tid & 15, by = tid >> 4, lane = tid & 31;
    const TileGeo g = tile_geo(P, tx, ty);
    const int W = P.W, rows = P.stack * P.tile_h;
    pkey_t *gk = P.keys;
    const int nrow = min(4, g.rv - 4 * by), ncol = min(4, g.wv - 4 * bx);
    pkey_t k[4][4];
    unsigned mine = 0;
    if (tid == 0) Q.n = 0;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const size_t o = (size_t)(g.y0 + 4 * by + r) * W + g.x0 + 4 * bx;
        load_keys(gk, o, r < nrow ? ncol : 0, (W & 1) == 0, k[r]);
    }
#pragma unroll
    for (int j = 0; j < 16; ++j)
        if (key_exits(k[j >> 2][j & 3])) mine |= 1u << j;
    __syncthreads();
    int pos = __popc(mine);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(FULL, pos, o);
        if (lane >= o) pos += v;
    }
    int base = 0;
    if (lane == 31) base = atomicAdd(&Q.n, pos);
    pos += __shfl_sync(FULL, base, 31) - __popc(mine);
#pragma unroll
    for (int j = 0; j < 16; ++j)
        if ((mine >> j) & 1u) {
            Q.key[pos] = k[j >> 2][j & 3];
            Q.at[pos++] = (unsigned short)((4 * by + (j >> 2)) * RT_COLS + 4 * bx + (j & 3));
        }
    __syncthreads();
    const int n = Q.n;
    for (int i0 = tid; i0 < n; i0 += NT * PER) {
        pkey_t kq[PER];
        int x0[PER], y0[PER];   // origins of the tiles that the chains have come to
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            kq[j] = i0 + j * NT < n ? Q.key[i0 + j * NT] : KEY_INF;
            x0[j] = g.x0;
            y0[j] = g.y0;
        }
        for (int step = 0; step < (1 << 20); ++step) {   // (distances fall: the bound is for form)
            bool more = false;
#pragma unroll
            for (int j = 0; j < PER; ++j)
                if (key_exits(kq[j])) {
                    const int cell = (int)key_label(kq[j]);
                    const int lr = cell / ROOT_PITCH - 1, lc = cell % ROOT_PITCH - 1;
                    kq[j] = __ldcg(gk + (size_t)(y0[j] + lr) * W + x0[j] + lc);
                    y0[j] += lr < 0 ? -rows : lr >= rows ? rows : 0;
                    x0[j] += lc < 0 ? -RT_COLS : lc >= RT_COLS ? RT_COLS : 0;
                    more = true;
                }
            if (!more) break;
        }
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            if (i0 + j * NT >= n) continue;
            const pkey_t own = Q.key[i0 + j * NT];
            const int at = Q.at[i0 + j * NT];
            gk[(size_t)(g.y0 + at / RT_COLS) * W + g.x0 + at % RT_COLS] =
                key_reached(kq[j]) ? (own & ~(FLAG | LABEL_NONE)) | key_label(kq[j]) : KEY_INF;
        }
    }
    __syncthreads();
}

// Calls f(P, tx, ty) for every tile this CTA owns.
template <typename F>
__device__ void each_tile(const BatchArgs &a, unsigned nblocks, F f) {
    for (unsigned t = blockIdx.x; t < (unsigned)a.total_solve; t += nblocks) {
        const int pi = find_pair(a.solve_base, a.npairs, (int)t);
        const PairDev &P = a.pairs[pi];
        const int lt = (int)t - a.solve_base[pi];
        f(P, lt % P.tiles_x, lt / P.tiles_x);
    }
}

// 384 threads per SM: the block's 16 distances and 86 weights, and the 20
// distances around it, take about 150 registers.
template <int MAXR>
__global__ void __launch_bounds__(Dim<MAXR>::NT, 384 / Dim<MAXR>::NT)
    relax_kernel(const BatchArgs *__restrict__ ap) {
    const BatchArgs a = *ap;
    RunState *st = a.state;
    if (get_status(st) != 0) return;  // same decision in every CTA
    // a launch replayed for a smaller batch may have more CTAs than tiles:
    // the extra CTAs leave at once
    const unsigned nblocks = min(gridDim.x, (unsigned)a.total_solve);
    if (blockIdx.x >= nblocks) return;
    __shared__ RelaxShared<MAXR> shared;
    DistTile<MAXR> &T = shared.dist;
    T.seeded[threadIdx.x] = 0;
    __syncthreads();

    // fresh, in two halves handed out by one counter: index u < T is tile
    // u of the first half (tx + ty even), index T + u tile u of the second.
    // Every first-half tile is taken before any second-half tile, so a
    // second-half tile only waits (bounded) for its four edge neighbours,
    // each already held by a running CTA; no grid barrier divides the
    // halves.
    for (;;) {
        if (threadIdx.x == 0) {
            int u;
            for (;;) {
                u = (int)atomicAdd(&st->work[3], 1u);
                if (u >= 2 * a.total_solve) break;
                const int half = u >= a.total_solve;
                const int t = u - (half ? a.total_solve : 0);
                const int pi = find_pair(a.solve_base, a.npairs, t);
                const int lt = t - a.solve_base[pi], TX = a.pairs[pi].tiles_x;
                if (((lt % TX + lt / TX) & 1) == half) break;
            }
            T.item = u;
        }
        __syncthreads();
        const int u = T.item;
        __syncthreads();
        if (u >= 2 * a.total_solve) break;
        const int half = u >= a.total_solve;
        const int t = u - (half ? a.total_solve : 0);
        const int pi = find_pair(a.solve_base, a.npairs, t);
        const PairDev &P = a.pairs[pi];
        const int lt = t - a.solve_base[pi];
        const int tx = lt % P.tiles_x, ty = lt / P.tiles_x;
        if (settles_only(P)) {
            seed_tile(P, lt, tx, ty, shared.root, st);
        } else {
            if (half && !wait_edge_neighbours(P, tx, ty, st)) return;
            solve_dist(P, lt, tx, ty, T, st, half ? SECOND : FIRST);
        }
        __syncthreads();
    }
    // spread: a tile or its ring may still be being written for the first time
    // when its owner comes to it, until all tiles are known to be written
    bool written = false;
    if (!own_tiles(a, st, &st->tiles[0], a.relax_req, T.own, nblocks,
              [&](const PairDev &P, int lt, int tx, int ty) -> unsigned {
                  if (settles_only(P)) return 0u;
                  if (!written) {
                      if (!wait_tile_and_ring(P, tx, ty, st)) return 0u;
                      written = __syncthreads_or(threadIdx.x == 0 && ld_acquire(&st->fresh_done) ==
                                                                         (unsigned)a.total_solve);
                  }
                  return solve_dist(P, lt, tx, ty, T, st, AGAIN);
              }))
        return;
    __syncthreads();
    each_tile(a, nblocks, [&](const PairDev &P, int tx, int ty) {
        if (!settles_only(P)) root_tile(P, tx, ty, T, shared.root, st);
    });
    __threadfence();
    if (!grid_sync(st, nblocks)) return;
    each_tile(a, nblocks, [&](const PairDev &P, int tx, int ty) {
        if (!settles_only(P)) chase_tile(P, tx, ty, shared.chase);
    });
    __threadfence();
    if (!grid_sync(st, nblocks)) return;
    if (!own_tiles(a, st, &st->tiles[1], a.relax_req + a.total_solve, shared.settle.own, nblocks,
                   [&](const PairDev &P, int, int tx, int ty) {
                       return settle_tile(P, tx, ty, shared.settle, st);
                   }))
        return;
    // nothing is left to do: report the re-solves as equivalent passes
    if (threadIdx.x == 0) {
        const unsigned long long Tt = (unsigned)a.total_solve;
        const unsigned long long n = (unsigned long long)ld_acquire(&st->tiles[0].solves) +
                                     ld_acquire(&st->tiles[1].solves);
        st->passes = (int)((n + Tt - 1) / Tt);
    }
}

// Self-test of this kernel's waits (see epic_selftest_wait_timeout): nothing
// stamps the tiles and nobody answers the request.
__device__ int selftest_words[4];
__global__ void relax_wait_selftest_kernel(RunState *st, int which, unsigned long long limit_ns) {
    __shared__ PairDev P;
    __shared__ OwnShared own;
    if (threadIdx.x == 0) {
        P.tiles_x = 2;   // two tiles side by side
        P.tiles_y = P.stack = 1;
        P.tile_stamp = selftest_words;
        selftest_words[0] = selftest_words[1] = STAMP_PENDING;
        selftest_words[2] = 0;   // requests of the one tile below
        st->tiles[0].open = 1;
    }
    __threadfence();
    __syncthreads();
    if (which == 2) {
        wait_edge_neighbours(P, 0, 0, st, limit_ns);
    } else if (which == 3) {
        wait_tile_and_ring(P, 0, 0, st, limit_ns);
    } else {
        BatchArgs a{};
        a.npairs = a.total_solve = a.total_tiles = a.max_passes = 1;
        own_tiles(a, st, &st->tiles[0], reinterpret_cast<unsigned *>(selftest_words + 2), own, 1u,
                  [](const PairDev &, int, int, int) { return 0u; }, limit_ns);
    }
}

}  // namespace

cudaError_t launch_relax_wait_selftest(RunState *st, int which, unsigned long long limit_ns, cudaStream_t stream) {
    relax_wait_selftest_kernel<<<1, 32, 0, stream>>>(st, which, limit_ns);
    return cudaGetLastError();
}

size_t relax_smem_bytes(int max_rows) {
    return max_rows <= 8    ? sizeof(RelaxShared<8>)
           : max_rows <= 16 ? sizeof(RelaxShared<16>)
                            : sizeof(RelaxShared<32>);
}

cudaError_t launch_relax(const BatchArgs &a, const BatchArgs *dev, const LaunchCfg &lc,
                         int max_rows, bool fixed_grid, int *grid_used) {
    if (max_rows < 1 || max_rows > RELAX_MAX_ROWS) return cudaErrorInvalidValue;
    // instances for tile heights up to 8, 16 and 32
    void (*kernel)(const BatchArgs *) = max_rows <= 8    ? relax_kernel<8>
                                        : max_rows <= 16 ? relax_kernel<16>
                                                         : relax_kernel<32>;
    const int threads = max_rows <= 8 ? Dim<8>::NT : max_rows <= 16 ? Dim<16>::NT : Dim<32>::NT;
    int grid = 0;
    cudaError_t e = launch_cooperative(kernel, threads, a.total_solve, fixed_grid, dev, lc, &grid);
    if (grid_used) *grid_used = grid;
    return e;
}

}  // namespace epic
