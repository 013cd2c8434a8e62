// Single-source geodesic distances of the exact variant: for every match, the
// distances of the pixels that can have it among their K nearest (those within
// their cap, see epic_exact_interp).
//
//   single_kernel  a CTA takes whole matches from a counter.  It holds keys
//                  of its own, a pool of tiles taken as a match touches them
//                  (a match that touches more is left for a second launch,
//                  with pools of every tile), and solves tiles of 64 x 32 pixels from the seed's outwards with the
//                  solve of relax_dist.cuh, the tile with the nearest open
//                  offer first: nothing passes between CTAs, so no fence,
//                  atomic or barrier of the grid is needed.  Only distances
//                  within the cap are written back; the cap is 1-Lipschitz in
//                  the same fixed-point metric, so every pixel on a shortest
//                  path to a pixel within its cap is within its own, and the
//                  capped distances are exact.  Pixels that can matter beyond
//                  a tile's 32-bit window are solved in further windows; what
//                  lies beyond 32 bits or MAX_WINDOWS, and every tile where the
//                  caps reach far (single_far in epic_internal.cuh), with 64-bit
//                  keys (relax_settle.cuh).  The tiles that a match reaches (13 of
//                  224 on a 1024 x 436 frame with 5000 matches and K = 100)
//                  are written out as float32 distance tiles.
//   cap_sum_kernel how far the caps reach.
//   map_tiles_kernel
//                  the distance tiles of matches that were relaxed by pairs (few
//                  matches, see epic_internal.cuh).
//   start_kernel,  the distance tiles by image tile, for the per-pixel fit.
//   list_kernel
//
// 1024 x 436, 5000 matches, K = 100: 11.5 ms; before, every match was a
// pseudo-pair of the apron-tile relaxation (directional sweeps in shared
// memory, a grid barrier per pass of a chunk of 300 matches) with a dense row
// of 446 K distances: 86.5 ms, and 5.3 ms to turn keys into rows.  What bounds
// it: the latency of a tile's rounds, with three CTAs a SM (registers).  45 solves and 52 windows per match, of ~10 K
// cycles for the rounds and ~14 K around them.  On the way to this form:
//   - 64-bit keys for a tile with any pixel beyond its window: 31 ms (half of
//     the solves, 91 K cycles each); further windows of 32 bits: 21.5 ms;
//   - nearest offer first and a window only when nothing nearer is open:
//     20.4 ms; offers tested against the ring's keys and caps, so that no
//     tile is asked that cannot use them (61 -> 45 solves): 16.2 ms.  First in,
//     first out instead: 19.0 ms; nearest by classes of 1/8 cost unit: 18.1;
//   - offers across windows from shared memory, for the pixels that need them
//     only, rather than unrolled in registers (41 K -> 20 K cycles): 13.9 ms;
//   - pools of tiles instead of a map of the frame per CTA, so that the budget
//     for keys (1 GiB) allows three CTAs a SM instead of two: 11.5 ms.
#include "relax_dist.cuh"
#include "relax_settle.cuh"

namespace epic {

namespace {

constexpr int SR = SINGLE_H;   // rows of a tile
constexpr int ST = Dim<SR>::NT;
constexpr int MAX_WINDOWS = 8;   // of a solve (1.2 on the flow workloads); beyond: 64-bit keys
constexpr int FEW = 512;         // frames of so many tiles (1 M pixels) have their tables in shared memory
constexpr unsigned char IN_QUEUE = 1, TOUCHED = 2;

// The tile with its ring, in image order, and the offers that lie beyond the
// window (for the next one).
struct WholeTile {
    unsigned d[SR + 2][RT_COLS + 2], h[SR + 2][RT_COLS + 2];
    unsigned far[16][ST];
};

struct SingleShared {
    union {
        struct {
            DistTile<SR> dist;
            WholeTile whole;
        };
        SettleTile<SR> settle;
    };
    ulonglong2 cap[8][ST];
    unsigned limit[RING<SR>];   // below what distance a ring pixel is improved
    unsigned offer[9];   // by neighbour (TB_*), and the tile itself: place of what is offered
    // the CTA's tiles (x.flags and so on), for frames of few tiles
    unsigned char flags[FEW];
    int queue[FEW], touched[FEW], place_of[FEW];
    unsigned at[FEW];
};

// The CTA's keys: a pool of tiles, taken in the order in which a match touches
// them.
struct PoolMap {
    pkey_t *pool, *own;    // own: of the tile being solved
    const int *place_of;   // tile -> place in the pool, -1: none (unreached)
    int tiles_x, x0, y0;
    __device__ __forceinline__ void row(int x, int y, int ncol, pkey_t *k) const {
        load_keys(own, (size_t)(y - y0) * SINGLE_W + x - x0, ncol, true, k);
    }
    __device__ __forceinline__ pkey_t at(int x, int y) const {
        const int s = place_of[y / SINGLE_H * tiles_x + x / SINGLE_W];
        return s < 0 ? KEY_INF
                     : __ldcg(pool + (size_t)s * SINGLE_TILE + y % SINGLE_H * SINGLE_W + x % SINGLE_W);
    }
};

// The distances and caps of this thread's ring pixels (unreached, 0: none).
constexpr int PER = (RING<SR> + ST - 1) / ST;
struct RingState {
    unsigned long long d[PER], cap[PER];
};
__device__ __forceinline__ void load_ring(const PairDev &P, const PoolMap &map, const pkey_t *cap, const TileGeo &g,
                                          RingState &R) {
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int i = threadIdx.x + j * ST;
        int lr, lc;
        ring_pixel<SR>(i, &lr, &lc);
        const int gx = g.x0 + lc, gy = g.y0 + lr;
        R.d[j] = ~0ull;
        R.cap[j] = 0;
        if (i < RING<SR> && lr <= g.rv && gx >= 0 && gx < P.W && gy >= 0 && gy < P.H) {
            const size_t o = (size_t)gy * P.W + gx;
            const pkey_t k = map.at(gx, gy);
            if (key_reached(k)) R.d[j] = key_dunits(k);
            R.cap[j] = key_dunits(cap[o]);
        }
    }
}
__device__ __forceinline__ void put_limits(const RingState &R, unsigned long long base, unsigned *limit) {
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int i = threadIdx.x + j * ST;
        const unsigned long long l = min(R.d[j], R.cap[j] + 1);
        if (i < RING<SR>) limit[i] = l <= base ? 0u : (unsigned)min(l - base, 0xFFFFFFFFull);
    }
}

// This thread's caps, fetched while its tile is staged and solved.
__device__ __forceinline__ void fetch_caps(const pkey_t *cap, const PairDev &P, const TileGeo &g,
                                           int nrow, int ncol, ulonglong2 (&to)[8][ST]) {
    const int tid = threadIdx.x, bx = tid & 15, by = tid >> 4;
    for (int r = 0; r < nrow; ++r) {
        const pkey_t *row = cap + (size_t)(g.y0 + 4 * by + r) * P.W + g.x0 + 4 * bx;
#pragma unroll
        for (int c = 0; c < 4; c += 2) {
            const unsigned s = (unsigned)__cvta_generic_to_shared(&to[2 * r + (c >> 1)][tid]);
            if (c + 1 < ncol && (P.W & 1) == 0)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(row + c) : "memory");
            else
                for (int i = c; i < min(c + 2, ncol); ++i)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(s + 8u * (i - c)), "l"(row + i)
                                 : "memory");
        }
    }
}
// (of cells outside the image: anything)
__device__ __forceinline__ void load_caps(const ulonglong2 (&from)[8][ST], unsigned long long (&v)[4][4]) {
    asm volatile("cp.async.wait_all;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const ulonglong2 k = from[i][threadIdx.x];
        v[i >> 1][2 * (i & 1)] = key_dunits(k.x);
        v[i >> 1][2 * (i & 1) + 1] = key_dunits(k.y);
    }
}

// A distance as a place in the queue.
__device__ __forceinline__ unsigned place(unsigned long long d) { return (unsigned)min(d >> 9, 0xFFFFFFFEull); }

__device__ __forceinline__ void store_row(pkey_t *dst, const pkey_t (&k)[4], unsigned mask, bool vec) {
    if (mask == 15u && vec) {
        reinterpret_cast<ulonglong2 *>(dst)[0] = make_ulonglong2(k[0], k[1]);
        reinterpret_cast<ulonglong2 *>(dst)[1] = make_ulonglong2(k[2], k[3]);
    } else {
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if ((mask >> c) & 1u) dst[c] = k[c];
    }
}

// The next window of a tile whose solve left `wanted` pixels unreached: the
// distances from S.base + S.win on.  Pixels below it are `known` and stand for
// its lower end; far holds, for every wanted pixel, the best offer of a known
// one (relative to S.base, exact: a step may be longer than a window).  Sets
// S.base, the block's distances (from the offers and the map) and the planes,
// and returns the sum that the map's distances alone would have (*before).
// false: nothing can be reached any more.  *lost: what matters lies beyond 32
// bits.
__device__ bool next_window(const PoolMap &map, const TileGeo &g, DistTile<SR> &T, WholeTile &A, DistBlock &B,
                            Staged &S, const RingState &R, unsigned known, unsigned wanted,
                            const ulonglong2 (&caps)[8][ST], unsigned long long *before, bool *lost) {
    const int tid = threadIdx.x, bx = tid & 15, by = tid >> 4;
    const int b = (by + 1) * RT_BX + bx + 1;
    const unsigned win = S.win;
    const unsigned long long base = S.base + win;
    auto rel = [&](unsigned long long d) -> unsigned {   // 0: below, 2^32 - 1: beyond 32 bits
        return d < base ? 0u : (unsigned)min(d - base, 0xFFFFFFFFull);
    };
    unsigned m = 0xFFFFFFFFu;   // the first distance of the window
    // whether a distance of the ring, of the map lies beyond 32 bits
    bool ring_beyond = false, map_beyond = false;
    int re[PER];
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int i = tid + j * ST;
        int lr, lc;
        ring_pixel<SR>(i, &lr, &lc);
        re[j] = i < RING<SR> ? plane_of(lr & 3, lc & 3) * Dim<SR>::NB + ring_entry(lr, lc) : -1;
        if (re[j] >= 0) {
            A.d[lr + 1][lc + 1] = (&T.d[0][0])[re[j]];
            A.h[lr + 1][lc + 1] = (&T.h[0][0])[re[j]];
            const unsigned rd = rel(R.d[j]);
            if (R.d[j] >= base) m = min(m, rd);
            ring_beyond |= rd == 0xFFFFFFFFu && R.d[j] != ~0ull;
        }
    }
    unsigned x[4][4];           // the map's
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        pkey_t k[4];
        map.row(g.x0 + 4 * bx, g.y0 + 4 * by + r, r < S.nrow ? S.ncol : 0, k);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            x[r][c] = key_reached(k[c]) ? rel(key_dunits(k[c])) : 0xFFFFFFFFu;
            if (!((known >> (4 * r + c)) & 1u)) {
                m = min(m, x[r][c]);
                map_beyond |= x[r][c] == 0xFFFFFFFFu && key_reached(k[c]);
            }
            A.d[4 * by + r + 1][4 * bx + c + 1] = B.d[r][c];
            A.h[4 * by + r + 1][4 * bx + c + 1] = S.h[r][c];
        }
    }
    __syncthreads();
#pragma unroll 1
    for (unsigned left = wanted; left; left &= left - 1) {
        // offers of the window before
        const int i = __ffs(left) - 1, y = 4 * by + (i >> 2), x = 4 * bx + (i & 3);
        const unsigned hp = A.h[y + 1][x + 1];
        unsigned long long best = 0xFFFFFFFFFFFFFFFFull;
#pragma unroll
        for (int n = 0; n < 9; ++n) {
            if (n == 4) continue;
            const unsigned q = A.d[y + n / 3][x + n % 3], hq = A.h[y + n / 3][x + n % 3];
            const unsigned long long w = (n & 1) ? (unsigned long long)hp + hq : step_diag(hp, hq);
            // (not negative: the pixel is outside the window)
            if (q < win) best = min(best, w - (win - q));
        }
        if (best > 0xFFFFFFFEull && best != 0xFFFFFFFFFFFFFFFFull)
            *lost |= base + best <= key_dunits(reinterpret_cast<const pkey_t *>(&caps[i >> 1][tid])[i & 1]);
        const unsigned old = A.far[i][tid] == 0xFFFFFFFFu ? 0xFFFFFFFFu : A.far[i][tid] - win;
        const unsigned f = min(old, (unsigned)min(best, 0xFFFFFFFFull));
        A.far[i][tid] = f;
        m = min(m, f);
    }
    m = __reduce_min_sync(FULL, m);
    if ((tid & 31) == 0) T.red[0][tid >> 5] = m;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < ST / 32; ++i) m = min(m, T.red[0][i]);
    // what lies beyond 32 bits of `base` may lie in the window, or be all there is
    *lost |= (map_beyond && m > 0xFFFFFFFFu - win) || (ring_beyond && m == 0xFFFFFFFFu);
    S.base = base + m;
    // (2^32 - 1, unreached or beyond 32 bits, is no distance)
    auto in = [&](unsigned d) { return d <= m ? 0u : d == 0xFFFFFFFFu ? win : min(d - m, win); };
    unsigned long long sum = 0;
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const bool below = (known >> (4 * r + c)) & 1u;
            sum += below ? win : in(x[r][c]);
            const bool held = (wanted >> (4 * r + c)) & 1u;   // (others: known, or their cap lies below)
            const unsigned far = held ? A.far[4 * r + c][tid] : 0xFFFFFFFFu;
            if (held && far != 0xFFFFFFFFu) A.far[4 * r + c][tid] = far - m;
            B.d[r][c] = below ? 0u : in(min(x[r][c], far));
            if (r == 0 || r == 3 || c == 0 || c == 3) T.d[plane_of(r, c)][b] = B.d[r][c];
        }
#pragma unroll
    for (int j = 0; j < PER; ++j)
        if (re[j] >= 0)
            (&T.d[0][0])[re[j]] = R.d[j] < S.base ? 0u : (unsigned)min(R.d[j] - S.base, (unsigned long long)win);
    *before = sum;
    bool more = false;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const ulonglong2 v = caps[i >> 1][tid];
        more |= ((wanted >> i) & 1u) && key_dunits(i & 1 ? v.y : v.x) >= S.base;
    }
    return __syncthreads_or(more) && m != 0xFFFFFFFFu;
}

// Solve tile (tx, ty) from the CTA's key map, window by window, and write back
// what lies within the cap.  sh.offer says what it offers its neighbours: the
// place of the nearest distance that can improve one of their pixels, 2^32 - 1
// for nothing (nothing within the cap changed; the match's first solve offers
// in any case, its seed is in the map already).  A window beyond `limit`, the
// first place in the queue, or beyond an offer waits: sh.offer[8].  far: with
// 64-bit keys at once.
__device__ void solve_single(const PairDev &P, const PoolMap &map, const pkey_t *cap, int tx, int ty, SingleShared &sh,
                             RunState *st, bool first, unsigned limit, bool far) {
    const int tid = threadIdx.x, bx = tid & 15, by = tid >> 4;
    const int b = (by + 1) * RT_BX + bx + 1;
    const TileGeo g = tile_geo(P, tx, ty);
    pkey_t *mine = map.own + 4 * by * SINGLE_W + 4 * bx;
    const int nrow = min(4, g.rv - 4 * by), ncol = min(4, g.wv - 4 * bx);
    bool wide = far;
    fetch_caps(cap, P, g, nrow, ncol, sh.cap);
    RingState R;
    if (!far) load_ring(P, map, cap, g, R);
    if (tid < 9) sh.offer[tid] = 0xFFFFFFFFu;   // (barriers follow)
    auto offer = [&](unsigned f, unsigned at) {
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if ((f >> k) & 1u) atomicMin(&sh.offer[k], at);
    };
    if (!far) {
        DistTile<SR> &T = sh.dist;
        DistBlock B;
        Staged S;
        stage_dist(P, tx, ty, g, T, B, S, st, AGAIN, map);
        block_weights(T, b, S, B);
        unsigned long long before = block_sum(B);
        unsigned known = 0;
        for (int window = 0;; ++window) {
            put_limits(R, S.base, sh.limit);
            dist_rounds(T, B, b, 2 + RT_COLS * SR);
            unsigned long long v[4][4];
            load_caps(sh.cap, v);
            unsigned wanted = 0, inside = 0;
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                pkey_t k[4];
                unsigned mask = 0;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const unsigned bit = 1u << (4 * r + c);
                    const bool fresh = r < nrow && c < ncol && !(known & bit);
                    const unsigned d = B.d[r][c];
                    const bool ok = fresh && d < S.win && S.base + d <= v[r][c];
                    // a pixel outside the window that its cap does not rule out
                    if (fresh && d >= S.win && v[r][c] >= S.base + S.win) wanted |= bit;
                    if (d < S.win) inside |= bit;
                    k[c] = make_key(S.base + d, LABEL_NONE);
                    if (ok) mask |= 1u << c;
                    else B.d[r][c] = S.win;
                }
                if (mask) store_row(mine + r * SINGLE_W, k, mask, true);
            }
            const bool changed = (first && window == 0) || block_sum(B) != before;
            if (__syncthreads_or(changed)) {
                const unsigned f = dist_offers(T, g, B, changed, sh.limit, S.win);
                if (f) {
                    unsigned d = S.win;
#pragma unroll
                    for (int i = 0; i < 16; ++i) d = min(d, B.d[i >> 2][i & 3]);
                    offer(f, place(S.base + d));
                }
            }
            if (!__syncthreads_or(wanted != 0)) break;
            const unsigned next = place(S.base + S.win);
            unsigned sooner = limit;
#pragma unroll
            for (int k = 0; k < 8; ++k) sooner = min(sooner, sh.offer[k]);
            if (next > sooner) {
                if (tid == 0) sh.offer[8] = next;
                break;
            }
            if (window == MAX_WINDOWS) {
                wide = true;
                break;
            }
            known |= inside;
            if (window == 0)
#pragma unroll
                for (int i = 0; i < 16; ++i) sh.whole.far[i][tid] = 0xFFFFFFFFu;
            bool lost = false;
            const bool more = next_window(map, g, T, sh.whole, B, S, R, known, wanted, sh.cap, &before, &lost);
            if (__syncthreads_or(lost)) {
                wide = true;
                break;
            }
            if (!more) break;
        }
    }
    if (wide) {
        SettleTile<SR> &T = sh.settle;
        Block B;
        stage_tile(P, T, g, B, st, map);
        const unsigned changed = solve_tile(T, g, B, st);
        unsigned long long v[4][4];
        load_caps(sh.cap, v);
        unsigned keep = 0;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            unsigned mask = 0;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int i = 4 * r + c;
                // (the seed, where no window has offered it yet)
                if (far && first && r < nrow && c < ncol && key_dunits(B.k[r][c]) == 0) keep |= 1u << i;
                if (!((changed >> i) & 1u) || r >= nrow || c >= ncol) continue;
                if (key_reached(B.k[r][c]) && key_dunits(B.k[r][c]) <= v[r][c]) mask |= 1u << c;
                else B.k[r][c] = KEY_INF;
            }
            if (mask) store_row(mine + r * SINGLE_W, B.k[r], mask, true);
            keep |= mask << (4 * r);
        }
        if (__syncthreads_or(keep != 0)) {
            const unsigned f = settle_offers(T, g, B, keep);
            if (f) {
                pkey_t k = KEY_INF;
#pragma unroll
                for (int i = 0; i < 16; ++i) k = min(k, B.k[i >> 2][i & 3]);
                offer(f, key_reached(k) ? place(key_dunits(k)) : 0u);
            }
        }
    }
    __syncthreads();
}

// Write the reached pixels of a tile, whose keys start at `keys` with `pitch` a
// row, out as a distance tile of match m.
__device__ void put_tile(const SingleArgs &x, int tile, const pkey_t *keys, int pitch, bool vec, int m,
                         int *shared_slot) {
    const int tid = threadIdx.x, bx = tid & 15, by = tid >> 4;
    const int rv = min(SINGLE_H, x.H - tile / x.tiles_x * SINGLE_H);
    const int wv = min(SINGLE_W, x.W - tile % x.tiles_x * SINGLE_W);
    const int nrow = min(4, rv - 4 * by), ncol = min(4, wv - 4 * bx);
    pkey_t k[4][4];
    bool any = false;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        load_keys(keys, (size_t)(4 * by + r) * pitch + 4 * bx, r < nrow ? ncol : 0, vec, k[r]);
#pragma unroll
        for (int c = 0; c < 4; ++c) any |= key_reached(k[r][c]);
    }
    if (!__syncthreads_or(any)) return;
    if (tid == 0) {
        const unsigned s = atomicAdd(x.used, 1u);
        *shared_slot = s < x.slot_cap ? (int)s : -1;
        if (s < x.slot_cap) {
            x.slot_of[s] = make_int2(tile, m);
            atomicAdd(x.tile_count + tile, 1);
        }
    }
    __syncthreads();
    const int s = *shared_slot;
#pragma unroll
    for (int r = 0; r < 4; ++r)
        if (s >= 0)
            *reinterpret_cast<float4 *>(x.slots + (size_t)s * SINGLE_TILE + (4 * by + r) * SINGLE_W + 4 * bx) =
                make_float4(key_dist(k[r][0]), key_dist(k[r][1]), key_dist(k[r][2]), key_dist(k[r][3]));
    __syncthreads();
}

// A CTA takes tile blockIdx.x of match m0 + blockIdx.y.
__global__ void __launch_bounds__(ST) map_tiles_kernel(SingleArgs x, const pkey_t *maps, int m0) {
    __shared__ int s_slot;
    const int tile = blockIdx.x;
    const size_t P = (size_t)x.H * x.W;
    const size_t at = blockIdx.y * P + (size_t)(tile / x.tiles_x * SINGLE_H) * x.W + tile % x.tiles_x * SINGLE_W;
    put_tile(x, tile, maps + at, x.W, (x.W & 1) == 0, m0 + (int)blockIdx.y, &s_slot);
}

// The sum of the distances of a map, in cost units (unreached: 1024).
__global__ void __launch_bounds__(256) cap_sum_kernel(const pkey_t *cap, long long n, float *sum) {
    float v = 0.f;
    for (long long i = blockIdx.x * 256LL + threadIdx.x; i < n; i += gridDim.x * 256LL)
        v += fminf(key_dist(cap[i]), 1024.f);
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
    __shared__ float s_part[8];
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) v += s_part[w];
        atomicAdd(sum, v);
    }
}

__global__ void __launch_bounds__(ST, 384 / ST) single_kernel(SingleArgs x) {
    RunState *st = x.state;
    const bool far = *x.cap_sum > x.cap_limit;
    if (get_status(st) != 0 || (x.far_returns && (far || *x.cap_sum < x.cap_floor))) return;
    __shared__ SingleShared sh;
    __shared__ PairDev P;
    __shared__ int s_item, s_queued, s_touched, s_slot, s_seed, s_fresh;
    __shared__ unsigned s_limit;
    const int tid = threadIdx.x;
    const int T = x.tiles_x * x.tiles_y;
    const bool few = T <= FEW;
    int *queue = few ? sh.queue : x.queue + (size_t)blockIdx.x * T;
    int *touched = few ? sh.touched : x.touched + (size_t)blockIdx.x * T;
    unsigned *at = few ? sh.at : x.place + (size_t)blockIdx.x * T;
    unsigned char *flags = few ? sh.flags : x.flags + (size_t)blockIdx.x * T;
    int *place_of = few ? sh.place_of : x.place_of + (size_t)blockIdx.x * T;
    PoolMap map{x.keys + (size_t)blockIdx.x * x.pool_tiles * SINGLE_TILE, nullptr, place_of, x.tiles_x, 0, 0};
    for (int i = tid; i < T; i += ST) {
        flags[i] = 0;
        place_of[i] = -1;
    }
    if (tid == 0) {
        P.C = x.C;
        P.matches = x.matches;
        P.H = x.H;
        P.W = x.W;
        P.tile_w = SINGLE_W;
        P.tile_h = SINGLE_H;
        P.stack = 1;
        P.tiles_x = x.tiles_x;
        P.tiles_y = x.tiles_y;
        P.sweep = 0;   // the unit 2^-31
    }
    __syncthreads();
    for (;;) {
        if (tid == 0) {
            const int i = (int)atomicAdd(x.next, 1u);
            const int m = i < x.N && x.list ? x.list[i] : i;
            s_item = i < x.N ? m : -1;
            s_queued = s_touched = 0;
            if (i < x.N) {
                const float4 mt = __ldg(x.matches + m);
                const float fx = floorf(mt.x + 0.5f), fy = floorf(mt.y + 0.5f);
                if (fx >= 0.f && fx < (float)x.W && fy >= 0.f && fy < (float)x.H) {
                    const int px = (int)fx, py = (int)fy;
                    const int t = py / SINGLE_H * x.tiles_x + px / SINGLE_W;
                    s_seed = py % SINGLE_H * SINGLE_W + px % SINGLE_W;
                    queue[s_queued++] = t;
                    at[t] = 0;
                    flags[t] = IN_QUEUE;
                } else {
                    set_status(st, EPIC_ERR_INVALID);
                }
            }
        }
        __syncthreads();
        const int m = s_item;
        __syncthreads();
        if (m < 0) return;
        bool whole = true;   // the pool held every tile that the match touches
        for (long long solves = 0;; ++solves) {
            // the nearest tile in the queue, and the place of the next one
            if (tid < 32) {
                const int n = s_queued;
                unsigned first = 0xFFFFFFFFu, second = 0xFFFFFFFFu;
                int fi = -1;
                for (int i = tid; i < n; i += 32) {
                    const unsigned p = at[queue[i]];
                    second = min(second, max(first, p));
                    if (p < first || fi < 0) {
                        first = p;
                        fi = i;
                    }
                }
                const unsigned best = __reduce_min_sync(FULL, first);
                const unsigned who = __ballot_sync(FULL, fi >= 0 && first == best);
                const bool mine = who && tid == __ffs(who) - 1;
                second = __reduce_min_sync(FULL, mine ? second : first);
                if (mine) {
                    const int t = queue[fi];
                    queue[fi] = queue[n - 1];
                    s_queued = n - 1;
                    s_fresh = 0;
                    s_item = t;
                    if (!(flags[t] & TOUCHED)) {
                        s_fresh = 1;
                        if (s_touched < x.pool_tiles) {
                            place_of[t] = s_touched;
                            touched[s_touched++] = t;
                        } else {
                            s_item = -2 - t;   // no room
                        }
                    }
                    flags[t] = TOUCHED;   // no longer queued
                    s_limit = second;
                }
                if (who == 0 && tid == 0) s_item = -1;
                if (tid == 0 && solves > x.max_solves) set_status(st, EPIC_ERR_NOT_CONVERGED);
            }
            __syncthreads();
            const int t = s_item;
            if (t < -1) whole = false;
            if (t < 0 || solves > x.max_solves) break;
            const int tx = t % x.tiles_x, ty = t / x.tiles_x;
            map.own = map.pool + (size_t)place_of[t] * SINGLE_TILE;
            map.x0 = tx * SINGLE_W;
            map.y0 = ty * SINGLE_H;
            if (s_fresh) {
                const pkey_t none[4] = {KEY_INF, KEY_INF, KEY_INF, KEY_INF};
                for (int i = 4 * tid; i < SINGLE_TILE; i += 4 * ST) store_row(map.own + i, none, 15u, true);
                __syncthreads();
                if (solves == 0 && tid == 0) map.own[s_seed] = make_key(0ull, LABEL_NONE);
                __syncthreads();
            }
            solve_single(P, map, x.cap, tx, ty, sh, st, solves == 0, s_limit, far);
            if (tid < 9 && sh.offer[tid] != 0xFFFFFFFFu) {
                const int nx = tid == 8 ? tx : tx + (tid < 3 ? tid - 1 : tid < 5 ? 2 * tid - 7 : tid - 6);
                const int ny = tid == 8 ? ty : ty + (tid < 3 ? -1 : tid < 5 ? 0 : 1);
                if (nx >= 0 && nx < x.tiles_x && ny >= 0 && ny < x.tiles_y) {
                    const int nt = ny * x.tiles_x + nx;
                    if (flags[nt] & IN_QUEUE) {
                        at[nt] = min(at[nt], sh.offer[tid]);
                    } else {
                        flags[nt] |= IN_QUEUE;
                        at[nt] = sh.offer[tid];
                        queue[atomicAdd(&s_queued, 1)] = nt;
                    }
                }
            }
            __syncthreads();
        }
        __syncthreads();
        const int n = s_touched;
        if (whole) {
            for (int i = 0; i < n; ++i)
                put_tile(x, touched[i], map.pool + (size_t)i * SINGLE_TILE, SINGLE_W, true, m, &s_slot);
        } else if (tid == 0) {
            x.left[atomicAdd(x.left_count, 1u)] = m;
            flags[-2 - s_item] = 0;
            for (int i = 0; i < s_queued; ++i) flags[queue[i]] = 0;
        }
        __syncthreads();
        for (int i = tid; i < n; i += ST) {
            flags[touched[i]] = 0;
            place_of[touched[i]] = -1;
        }
        __syncthreads();
    }
}

// One CTA: offsets of the image tiles' lists (tile_count becomes the cursor).
__global__ void __launch_bounds__(1024) start_kernel(int *count, int *start, int T) {
    __shared__ int warp_sums[32], carry;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (tid == 0) carry = 0;
    __syncthreads();
    for (int base = 0; base < T; base += 1024) {
        const int v = base + tid < T ? count[base + tid] : 0;
        int s = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(FULL, s, o);
            if (lane >= o) s += u;
        }
        if (lane == 31) warp_sums[wid] = s;
        __syncthreads();
        if (wid == 0) {
            int u = warp_sums[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int w = __shfl_up_sync(FULL, u, o);
                if (lane >= o) u += w;
            }
            warp_sums[lane] = u;
        }
        __syncthreads();
        const int at = carry + s - v + (wid ? warp_sums[wid - 1] : 0);
        if (base + tid < T) {
            start[base + tid] = at;
            count[base + tid] = at;
        }
        __syncthreads();
        if (tid == 1023) carry = at + v;
        __syncthreads();
    }
    if (tid == 0) start[T] = carry;
}

__global__ void list_kernel(SingleArgs x, unsigned used) {
    for (unsigned s = blockIdx.x * blockDim.x + threadIdx.x; s < used; s += gridDim.x * blockDim.x) {
        const int2 e = x.slot_of[s];
        x.tile_entry[atomicAdd(x.tile_count + e.x, 1)] = make_int2(e.y, (int)s);
    }
}

}  // namespace

int single_resident(int num_sms) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, single_kernel, ST, 0) != cudaSuccess ||
        per_sm < 1)
        per_sm = 1;
    return per_sm * num_sms;
}

cudaError_t launch_single(const SingleArgs &x, int ctas, cudaStream_t stream) {
    single_kernel<<<ctas, ST, 0, stream>>>(x);
    return cudaGetLastError();
}

cudaError_t launch_cap_sum(const pkey_t *cap, long long n, float *sum, cudaStream_t stream) {
    const cudaError_t e = cudaMemsetAsync(sum, 0, sizeof(float), stream);
    if (e != cudaSuccess) return e;
    const long long blocks = (n + 1023) / 1024;
    cap_sum_kernel<<<(unsigned)(blocks < 1024 ? blocks : 1024), 256, 0, stream>>>(cap, n, sum);
    return cudaGetLastError();
}

cudaError_t launch_map_tiles(const SingleArgs &x, const pkey_t *maps, int m0, int n, cudaStream_t stream) {
    const size_t P = (size_t)x.H * x.W;
    for (int j = 0; j < n; j += 65535) {   // (the grid's rows)
        const dim3 grid((unsigned)(x.tiles_x * x.tiles_y), (unsigned)(n - j < 65535 ? n - j : 65535));
        map_tiles_kernel<<<grid, ST, 0, stream>>>(x, maps + j * P, m0 + j);
    }
    return cudaGetLastError();
}

cudaError_t launch_single_lists(const SingleArgs &x, unsigned used, cudaStream_t stream) {
    start_kernel<<<1, 1024, 0, stream>>>(x.tile_count, x.tile_start, x.tiles_x * x.tiles_y);
    const unsigned blocks = (used + 255) / 256;
    list_kernel<<<blocks < 1 ? 1 : blocks < 1024 ? blocks : 1024, 256, 0, stream>>>(x, used);
    return cudaGetLastError();
}

}  // namespace epic
