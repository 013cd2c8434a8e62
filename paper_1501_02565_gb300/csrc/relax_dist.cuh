// The relaxation's distances: the geodesic distance D of every pixel to its
// nearest match, solved tile by tile (see k_relax.cu).
//
// A tile is 64 columns x up to R rows (R = 8, 16 or 32: a kernel instance
// each), solved by one CTA.  A thread holds a block of 4 x 4 pixels and the
// weights of all its steps in registers; a round of the solve is
//
//   forward   the block's pixels in raster order, each from its left, upper
//             left, upper and upper right neighbour;
//   backward  the same pixels in the opposite order from the other four;
//
// with the 20 distances around the block read from shared memory before and
// its 12 border distances written back after.  The rounds end when one
// changes nothing.  A distance crosses a whole block per round, so a fresh
// tile of the flow workloads takes ~9 rounds and a re-solve ~2.3, with every
// pixel of the tile busy in each.
//
// Only distances are carried, as 32-bit words relative to the tile's smallest:
// a step is then one add-and-minimum (VIADDMNMX), half a cycle per warp and
// SM, where a step that carries the packed 64-bit (D, L) key takes 2.6 (an
// IMAD.WIDE, a 64-bit compare and select; measured).  A tile's words span the
// window [0, T), T = 2^31 - 1 at most: a distance beyond it (1.0 cost units
// above the tile's smallest, a pixel inside a strong edge) is left unreached
// here, and so is nothing else, because a path to a pixel inside the window
// never leaves it.  The settling pass completes those pixels: it
// takes any map of upper bounds to the exact fixed point.
//
// Shared-memory layout: plane q holds border cell q of every block, one entry
// per block with a ring of blocks around the tile for its outer pixels.  The
// lanes of a warp (two rows of 16 blocks) then always read and write
// consecutive entries: no bank conflicts.
#pragma once

#include "relax_tiles.cuh"

namespace epic {

namespace {

template <int MAXR>
struct DistTile {
    using D = Dim<MAXR>;
    unsigned d[12][D::NB];     // border distances of every block (and of the ring's)
    unsigned h[12][D::NB];     // border half-costs
    unsigned seeded[D::NT];    // cells of a block that hold a seed
    unsigned red[2][D::NT / 32];
    unsigned flags;            // what the solve did (TB_*)
    int item;                  // broadcast of thread 0's choice
    OwnShared own;
};

// A thread's block: distances relative to the tile's base (T: not in the
// window), and the weights of its steps: wh[r][c] between columns c - 1 and c
// of row r, wv[r][c] between rows r - 1 and r of column c, wb[r][c] between
// (r - 1, c - 1) and (r, c), ws[r][c] between (r - 1, c) and (r, c - 1).
struct DistBlock {
    unsigned d[4][4];
    unsigned wh[4][5], wv[5][4], wb[5][5], ws[5][5];
};

// How a tile is staged and solved: FIRST and SECOND are the halves of phase 1,
// AGAIN a phase-2 solve from the current key map, ROOT the look for parents.
enum Mode { FIRST, SECOND, AGAIN, ROOT };

// What a thread keeps of a staging besides its block.
struct Staged {
    unsigned h[4][4];          // half-costs
    unsigned long long base;   // the tile's smallest distance (rounded down)
    unsigned win;              // the window: distances in [base, base + win)
    int nrow, ncol;            // of the block inside the image (and the ring row)
};

// A key whose pixel is rooted outside its tile, until the chains are followed
// (see k_relax.cu): the unreached flag, the distance (not zero: a parent is
// strictly nearer) and, in place of the label, the cell of the tile's ring
// that the pixel's path leads to.
constexpr pkey_t FLAG = 0x8000000000000000ull;
__device__ __forceinline__ bool key_exits(pkey_t k) { return (k & FLAG) && key_dunits(k & ~FLAG); }
// A key of the map without its label, whatever the look for parents has done.
__device__ __forceinline__ pkey_t bare_key(pkey_t k) {
    return (key_exits(k) ? k & ~FLAG : k) | LABEL_NONE;
}

// min(round(sqrt(2) (h_p + h_q)), cap): step_diag, capped
__device__ __forceinline__ unsigned diag_weight(unsigned hp, unsigned hq, unsigned cap) {
    const unsigned long long x = (unsigned long long)(hp + hq) * SQRT2_Q30 + (1ull << 29);
    const unsigned hi = (unsigned)(x >> 32);
    const unsigned w = __funnelshift_r((unsigned)x, hi, 30);
    return hi >= (1u << 30) ? cap : min(w, cap);
}

__device__ __forceinline__ void lower(unsigned &d, unsigned q, unsigned w) {
    d = __viaddmin_u32(q, w, d);
}

// The sum of a block's distances, which only fall, so that it changes whenever
// one does.
__device__ __forceinline__ unsigned long long block_sum(const DistBlock &B) {
    unsigned long long s = 0;
#pragma unroll
    for (int i = 0; i < 16; ++i)   // (IMAD.WIDE: not on the integer pipe)
        asm("mad.wide.u32 %0, %1, 1, %0;" : "+l"(s) : "r"(B.d[i >> 2][i & 3]));
    return s;
}

// The rounds of a solve.
template <int MAXR>
__device__ void dist_rounds(DistTile<MAXR> &T, DistBlock &B, int b, int cap) {
    unsigned long long sum = block_sum(B);
    for (int round = 0; round < cap; ++round) {
        unsigned w[4], e[4], n[6], s[6];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            w[r] = around(T.d, b, r, -1);
            e[r] = around(T.d, b, r, 4);
        }
#pragma unroll
        for (int c = 0; c < 6; ++c) n[c] = around(T.d, b, -1, c - 1);
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                unsigned d = B.d[r][c];
                lower(d, r ? B.d[r - 1][c] : n[c + 1], B.wv[r][c]);
                lower(d, r ? (c ? B.d[r - 1][c - 1] : w[r - 1]) : n[c], B.wb[r][c]);
                lower(d, r ? (c < 3 ? B.d[r - 1][c + 1] : e[r - 1]) : n[c + 2], B.ws[r][c + 1]);
                lower(d, c ? B.d[r][c - 1] : w[r], B.wh[r][c]);
                B.d[r][c] = d;
            }
#pragma unroll
        for (int c = 0; c < 6; ++c) s[c] = around(T.d, b, 4, c - 1);
#pragma unroll
        for (int r = 3; r >= 0; --r)
#pragma unroll
            for (int c = 3; c >= 0; --c) {
                unsigned d = B.d[r][c];
                lower(d, r < 3 ? B.d[r + 1][c] : s[c + 1], B.wv[r + 1][c]);
                lower(d, r < 3 ? (c < 3 ? B.d[r + 1][c + 1] : e[r + 1]) : s[c + 2], B.wb[r + 1][c + 1]);
                lower(d, r < 3 ? (c ? B.d[r + 1][c - 1] : w[r + 1]) : s[c], B.ws[r + 1][c]);
                lower(d, c < 3 ? B.d[r][c + 1] : e[r], B.wh[r][c + 1]);
                B.d[r][c] = d;
            }
        const unsigned long long now = block_sum(B);
        const bool changed = now != sum;
        sum = now;
        if (changed) {
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (r == 0 || r == 3 || c == 0 || c == 3) T.d[plane_of(r, c)][b] = B.d[r][c];
        }
        if (!__syncthreads_or(changed)) break;
    }
}

// Stage tile (tx, ty): this thread's distances into B.d and the rest into S,
// the tile's border distances and half-costs and the ring into shared memory;
// every thread has passed a barrier when it returns.
template <int MAXR, typename Map = FrameMap>
__device__ void stage_dist(const PairDev &P, int tx, int ty, const TileGeo &g, DistTile<MAXR> &T,
                           DistBlock &B, Staged &S, RunState *st, Mode mode, const Map &map) {
    constexpr int NT = Dim<MAXR>::NT, NB = Dim<MAXR>::NB;
    const int tid = threadIdx.x, bx = tid & 15, by = tid >> 4;
    const int b = (by + 1) * RT_BX + bx + 1;
    const int W = P.W, H = P.H;
    const float *gc = P.C;
    const bool cvec = (W & 3) == 0 && ((uintptr_t)gc & 15) == 0;

    // this block's costs and keys (rows down to the ring row below the tile,
    // which lies inside a block when the tile is not a whole number of blocks
    // high: it is solved along, and not written), and its share of the ring
    const int nrow = S.nrow = min(4, min(g.rv + 1, H - g.y0) - 4 * by);
    const int ncol = S.ncol = min(4, g.wv - 4 * bx);
    float cc[4][4];
    pkey_t kk[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const size_t o = (size_t)(g.y0 + 4 * by + r) * W + g.x0 + 4 * bx;
        const int nc = r < nrow ? ncol : 0;
        load_costs(gc, o, nc, cvec, cc[r]);
        const bool ring_row = 4 * by + r >= g.rv;
        map.row(g.x0 + 4 * bx, g.y0 + 4 * by + r, mode >= AGAIN || (mode == SECOND && ring_row) ? nc : 0, kk[r]);
    }
    constexpr int PER = (RING<MAXR> + NT - 1) / NT;
    pkey_t rk[PER];
    float rc[PER];
    int re[PER];   // plane entry, -1: nothing
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int i = tid + j * NT;
        int lr, lc;
        ring_pixel<MAXR>(i, &lr, &lc);
        re[j] = i < RING<MAXR> ? plane_of(lr & 3, lc & 3) * NB + ring_entry(lr, lc) : -1;
        const int gx = g.x0 + lc, gy = g.y0 + lr;
        const bool in = i < RING<MAXR> && lr <= g.rv && gx >= 0 && gx < W && gy >= 0 && gy < H;
        const bool diagonal = (lr < 0 || lr >= g.rv) && (lc < 0 || lc >= RT_COLS);
        rk[j] = KEY_INF;
        rc[j] = 0.f;
        if (in) {
            const size_t o = (size_t)gy * W + gx;
            rc[j] = __ldg(gc + o);
            if (mode >= AGAIN || (mode == SECOND && !diagonal)) rk[j] = map.at(gx, gy);
        }
    }
    if (mode == ROOT) {
        // the tiles next door may carry their labels already
#pragma unroll
        for (int j = 0; j < PER; ++j) rk[j] = bare_key(rk[j]);
#pragma unroll
        for (int i = 0; i < 16; ++i) kk[i >> 2][i & 3] = bare_key(kk[i >> 2][i & 3]);
    }
    unsigned lo = 0xFFFFFFFFu;   // smallest distance, in units of 2^9
    if (mode < AGAIN) {
        // the seeds of the stacked tiles' bins (the masks are zero between solves)
        for (int q = 0; q < P.stack && ty * P.stack + q < P.tiles_y; ++q) {
            const int bin = (ty * P.stack + q) * P.tiles_x + tx;
            for (int s = P.tile_start[bin] + tid, s1 = P.tile_start[bin + 1]; s < s1; s += NT) {
                const float4 mt = __ldg(P.matches + P.tile_seeds[s]);
                const int px = (int)floorf(mt.x + 0.5f) - g.x0;
                const int py = (int)floorf(mt.y + 0.5f) - g.y0;
                if (px >= 0 && px < g.wv && py >= 0 && py < g.rv) {
                    atomicOr(&T.seeded[(py >> 2) * 16 + (px >> 2)], 1u << (4 * (py & 3) + (px & 3)));
                    lo = 0;
                }
            }
        }
    }
    HalfCost half(P);
    auto coarse = [](pkey_t k) { return key_reached(k) ? (unsigned)(k >> (LABEL_BITS + 9)) : 0xFFFFFFFFu; };
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            S.h[r][c] = half(cc[r][c]);
            lo = min(lo, coarse(kk[r][c]));
            if (r == 0 || r == 3 || c == 0 || c == 3) T.h[plane_of(r, c)][b] = S.h[r][c];
        }
#pragma unroll
    for (int j = 0; j < PER; ++j)
        if (re[j] >= 0) {
            (&T.h[0][0])[re[j]] = half(rc[j]);
            lo = min(lo, coarse(rk[j]));
        }
    if (half.bad) set_status(st, EPIC_ERR_INVALID);
    lo = __reduce_min_sync(FULL, lo);
    unsigned hm = __reduce_max_sync(FULL, half.largest);
    if ((tid & 31) == 0) {
        T.red[0][tid >> 5] = lo;
        T.red[1][tid >> 5] = hm;
    }
    if (tid == 0) T.flags = 0;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NT / 32; ++i) {
        lo = min(lo, T.red[0][i]);
        hm = max(hm, T.red[1][i]);
    }
    // The window: T + 2 hm < 2^32, so that no candidate overflows, and
    // diagonal weights are capped at 2^32 - 1 - T >= T, which never offers a
    // distance inside the window.
    const unsigned long long base = S.base = lo == 0xFFFFFFFFu ? 0ull : (unsigned long long)lo << 9;
    const unsigned win = S.win = min(0x7FFFFFFFu, 0xFFFFFFFFu - 2u * hm);
    auto rel = [&](pkey_t k) -> unsigned {
        const unsigned long long x = key_dunits(k) - base;
        return key_reached(k) && x < win ? (unsigned)x : win;
    };
#pragma unroll
    for (int j = 0; j < PER; ++j)
        if (re[j] >= 0) (&T.d[0][0])[re[j]] = rel(rk[j]);
    unsigned seeds = 0;
    if (mode < AGAIN) {
        seeds = T.seeded[tid];
        T.seeded[tid] = 0;
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            B.d[r][c] = (seeds >> (4 * r + c)) & 1u ? 0u : rel(kk[r][c]);
            if (r == 0 || r == 3 || c == 0 || c == 3) T.d[plane_of(r, c)][b] = B.d[r][c];
        }
    __syncthreads();
}

// The weights of a staged block's steps.
template <int MAXR>
__device__ void block_weights(const DistTile<MAXR> &T, int b, const Staged &S, DistBlock &B) {
    const unsigned wmax = 0xFFFFFFFFu - S.win;
    auto hc = [&](int r, int c) {
        return r >= 0 && r < 4 && c >= 0 && c < 4 ? S.h[r & 3][c & 3] : around(T.h, b, r, c);
    };
    // weights; a step to a cell of the block that lies outside the image
    // (or below the ring row) is blocked by the cap
    unsigned hr[6][6];
#pragma unroll
    for (int r = 0; r < 6; ++r)
#pragma unroll
        for (int c = 0; c < 6; ++c) hr[r][c] = hc(r - 1, c - 1);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            B.wh[i][j] = hr[i + 1][j] + hr[i + 1][j + 1];
            B.wv[j][i] = hr[j][i + 1] + hr[j + 1][i + 1];
        }
#pragma unroll
    for (int r = 0; r < 5; ++r)
#pragma unroll
        for (int c = 0; c < 5; ++c) {
            if (!((r == 0 && c == 4) || (r == 4 && c == 0)))
                B.wb[r][c] = diag_weight(hr[r][c], hr[r + 1][c + 1], wmax);
            if (!((r == 0 && c == 0) || (r == 4 && c == 4)))
                B.ws[r][c] = diag_weight(hr[r][c + 1], hr[r + 1][c], wmax);
        }
    if (S.nrow < 4 || S.ncol < 4) {
        auto out = [&](int r, int c) {   // own cells only: the ring's are never lowered
            return r >= 0 && r < 4 && c >= 0 && c < 4 && (r >= S.nrow || c >= S.ncol);
        };
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 5; ++j) {
                if (out(i, j - 1) || out(i, j)) B.wh[i][j] = wmax;
                if (out(j - 1, i) || out(j, i)) B.wv[j][i] = wmax;
            }
#pragma unroll
        for (int r = 0; r < 5; ++r)
#pragma unroll
            for (int c = 0; c < 5; ++c) {
                if (out(r - 1, c - 1) || out(r, c)) B.wb[r][c] = wmax;
                if (out(r - 1, c) || out(r, c - 1)) B.ws[r][c] = wmax;
            }
    }
}

// Which neighbours' border pixels this thread's border pixels improve (TB_*
// bits).  changed: the block has changed (for a ring row that lies among the
// blocks: any change of the last row's).  limit: below what distance each ring
// pixel is improved (in ring_pixel's order); without it, below the staged one
// (pixels outside the window are left to the settling pass).
template <int MAXR>
__device__ unsigned dist_offers(const DistTile<MAXR> &T, const TileGeo &g, const DistBlock &B,
                                bool changed, const unsigned *limit = nullptr, unsigned win = 0) {
    const int tid = threadIdx.x, bx = tid & 15, by = tid >> 4;
    const int b = (by + 1) * RT_BX + bx + 1;
    unsigned f = 0;
    auto offers = [&](int r, int c, int r2, int c2, unsigned w) {
        if (!limit) return B.d[r][c] + w < around(T.d, b, r2, c2);
        const int lr = 4 * by + r2, lc = 4 * bx + c2;
        const int i = r2 < 0 && by == 0 ? lc + 1
                      : r2 > 3 && lr == MAXR ? RT_COLS + 2 + lc + 1
                                             : 2 * (RT_COLS + 2) + 2 * lr + (c2 > 0 ? 1 : 0);
        return B.d[r][c] < win && B.d[r][c] + w < limit[i];
    };
    bool up = false, down = false, left = false, right = false;
    if (by == 0) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            up |= offers(0, c, -1, c, B.wv[0][c]);
            if (c || bx) up |= offers(0, c, -1, c - 1, B.wb[0][c]);
            if (c < 3 || bx < 15) up |= offers(0, c, -1, c + 1, B.ws[0][c + 1]);
        }
        if (bx == 0 && offers(0, 0, -1, -1, B.wb[0][0])) f |= TB_UL;
        if (bx == 15 && offers(0, 3, -1, 4, B.ws[0][4])) f |= TB_UR;
    }
    if (g.rv == MAXR) {
        if (4 * by + 4 == MAXR) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                down |= offers(3, c, 4, c, B.wv[4][c]);
                if (c < 3 || bx < 15) down |= offers(3, c, 4, c + 1, B.wb[4][c + 1]);
                if (c || bx) down |= offers(3, c, 4, c - 1, B.ws[4][c]);
            }
            if (bx == 0 && offers(3, 0, 4, -1, B.ws[4][0])) f |= TB_DL;
            if (bx == 15 && offers(3, 3, 4, 4, B.wb[4][4])) f |= TB_DR;
        }
    } else if (changed && 4 * by < g.rv && 4 * by + 4 >= g.rv) {
        // the ring row lies among the blocks: any change of the last row's
        f |= TB_D | (bx == 0 ? TB_DL : 0u) | (bx == 15 ? TB_DR : 0u);
    }
    if (bx == 0) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            left |= offers(r, 0, r, -1, B.wh[r][0]);
            if (r || by) left |= offers(r, 0, r - 1, -1, B.wb[r][0]);
            if (4 * by + r + 1 < g.rv) left |= offers(r, 0, r + 1, -1, B.ws[r + 1][0]);
        }
    }
    if (bx == 15) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            right |= offers(r, 3, r, 4, B.wh[r][4]);
            if (r || by) right |= offers(r, 3, r - 1, 4, B.ws[r][4]);
            if (4 * by + r + 1 < g.rv) right |= offers(r, 3, r + 1, 4, B.wb[r + 1][4]);
        }
    }
    return f | (up ? TB_U : 0u) | (down ? TB_D : 0u) | (left ? TB_L : 0u) | (right ? TB_R : 0u);
}

// Solve tile (tx, ty), local index t.
//   FIRST   alone, from its own seeds, with an unreached ring;
//   SECOND  from its seeds and the ring of its four edge neighbours, solved
//           by then (pixels of the diagonal neighbours, which belong to tiles
//           of the same half, stay unreached);
//   AGAIN   from its current keys and the ring's.
// The first two write every key of the tile, AGAIN a changed tile's.  Keys
// carry no label yet.
// Returns, in every thread, what the solve did (TB_*; 0: nothing changed).
template <int MAXR>
__device__ unsigned solve_dist(const PairDev &P, int t, int tx, int ty, DistTile<MAXR> &T,
                               RunState *st, Mode mode) {
    const int tid = threadIdx.x, bx = tid & 15, by = tid >> 4;
    const int b = (by + 1) * RT_BX + bx + 1;
    const TileGeo g = tile_geo(P, tx, ty);
    const int W = P.W;
    DistBlock B;
    Staged S;
    stage_dist(P, tx, ty, g, T, B, S, st, mode, FrameMap(P));
    unsigned f = mode != AGAIN ? TB_ANY : 0u;
    {
        block_weights(T, b, S, B);
        const unsigned long long before = block_sum(B);   // (cells below the tile count, harmlessly)
        dist_rounds(T, B, b, 2 + RT_COLS * MAXR);
        const unsigned long long after = block_sum(B);
        if (before != after) f |= TB_ANY;
        if (mode == AGAIN && __syncthreads_or(before != after)) {
            f |= dist_offers(T, g, B, before != after);
        }
    }
    if (f & TB_ANY) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            if (4 * by + r >= g.rv || r >= S.nrow) continue;
            pkey_t *dst = P.keys + (size_t)(g.y0 + 4 * by + r) * W + g.x0 + 4 * bx;
            pkey_t k[4];
            bool all = S.ncol >= 4 && (W & 1) == 0;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                // (a distance beyond the 41 bits of a key is left unreached too)
                const bool in = B.d[r][c] < S.win && S.base + B.d[r][c] < (1ull << 41);
                k[c] = in ? make_key(S.base + B.d[r][c], LABEL_NONE) : KEY_INF;
                all = all && (in || mode != AGAIN);
            }
            if (all) {
                reinterpret_cast<ulonglong2 *>(dst)[0] = make_ulonglong2(k[0], k[1]);
                reinterpret_cast<ulonglong2 *>(dst)[1] = make_ulonglong2(k[2], k[3]);
            } else {
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (c < S.ncol && (mode != AGAIN || key_reached(k[c]))) dst[c] = k[c];
            }
        }
        if (mode != AGAIN) __threadfence();   // (own_tiles fences an AGAIN solve)
    }
    f = __reduce_or_sync(FULL, f);
    if (f && (tid & 31) == 0) atomicOr(&T.flags, f);
    __syncthreads();
    f = T.flags;
    if (!(f & TB_ANY)) return 0;
    if (mode != AGAIN && tid == 0) {
        *(volatile int *)(P.tile_stamp + t) = 0;
        __threadfence();
        atomicAdd(&st->fresh_done, 1u);
    }
    return f;
}

}  // namespace

}  // namespace epic
