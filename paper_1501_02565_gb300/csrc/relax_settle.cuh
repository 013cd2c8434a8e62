// The relaxation's last pass: the packed (D, L) keys are relaxed to their
// fixed point, tile by tile (see k_relax.cu).
//
// A solve is built like that of the distances (relax_dist.cuh): 4 x 4 pixels
// a thread, forward and backward sweeps.  It carries whole keys, though: a
// candidate is an IMAD.WIDE (the key plus weight x 2^22, on the FMA pipe), a
// 64-bit compare and a 64-bit select, 2.6 cycles per warp and SM.
#pragma once

#include "relax_tiles.cuh"

namespace epic {

namespace {

constexpr int DIAG_EDGES = 46;  // diagonal steps with an end in a block

// The settling relaxation's tile.  The weights of a block's diagonal steps
// are computed once per solve and kept in shared memory, in the space of the
// half-cost planes, which only their computation needs.
template <int MAXR>
struct SettleTile {
    using D = Dim<MAXR>;
    pkey_t K[12][D::NB];                // border keys of every block (and of the ring's)
    union {
        unsigned h[12][D::NB];          // border half-costs, while a tile is staged
        unsigned wd[DIAG_EDGES][D::NT]; // diagonal weights of a thread's block
    };
    unsigned hmax[D::NT / 32];
    unsigned flags;                     // what the solve did (TB_*)
    int big;                            // diagonal weights need more than 32 bits
    OwnShared own;
};
__device__ __forceinline__ pkey_t kmin(pkey_t a, pkey_t b) { return b < a ? b : a; }

// kq + (w << LABEL_BITS) as one IMAD.WIDE
__device__ __forceinline__ pkey_t key_plus(pkey_t kq, unsigned w) {
    pkey_t r;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(w), "r"(1u << LABEL_BITS), "l"(kq));
    return r;
}

// the axis step from q: two IMAD.WIDE.  (Adding h_p + h_q first would take
// the busier pipe, and the compiler would keep all 40 sums of a block in
// registers across the rounds and spill the keys.)
__device__ __forceinline__ pkey_t key_axis(pkey_t kq, unsigned hp, unsigned hq) {
    return key_plus(key_plus(kq, hq), hp);
}

// index of the weight of a block's diagonal step from (r, c): to the upper
// left, upper right, lower left, lower right
__host__ __device__ constexpr int e_ul(int r, int c) { return 4 * r + c; }
__host__ __device__ constexpr int e_ur(int r, int c) { return 16 + 4 * r + c; }
__host__ __device__ constexpr int e_ll(int r, int c) {
    return r < 3 && c > 0 ? e_ur(r + 1, c - 1) : r == 3 ? 32 + c : 36 + r;
}
__host__ __device__ constexpr int e_lr(int r, int c) {
    return r < 3 && c < 3 ? e_ul(r + 1, c + 1) : r == 3 ? 39 + c : 43 + r;
}

// A thread's block: keys, half-costs, and the half-costs above, below, left
// and right of it.
struct Block {
    pkey_t k[4][4];
    unsigned h[4][4];
    unsigned hn[4], hs[4], hw[4], he[4];
    unsigned valid;   // bit 4 r + c: the cell is a pixel of the tile
};

// The rounds of a solve.  FULL_TILE: every cell of every block is a pixel of
// the tile.  BIG: some diagonal weight of the tile needs more than 32 bits
// (costs above 1.41 units), so the weights are formed at every use.  Returns
// the mask of this thread's changed cells.
template <int MAXR, bool FULL_TILE, bool BIG>
__device__ unsigned rounds(SettleTile<MAXR> &T, Block &B, int b, int cap, RunState *st) {
    const int tid = threadIdx.x;
    unsigned changed = 0;
    auto diag = [&](pkey_t kq, int e, unsigned hp, unsigned hq) -> pkey_t {
        return BIG ? step_key(kq, step_diag(hp, hq)) : key_plus(kq, T.wd[e][tid]);
    };
    for (int round = 0;; ++round) {
        unsigned now = 0;
        pkey_t w[4], e[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            w[r] = around(T.K, b, r, -1);
            e[r] = around(T.K, b, r, 4);
        }
        {
            pkey_t n[6];
#pragma unroll
            for (int c = 0; c < 6; ++c) n[c] = around(T.K, b, -1, c - 1);
            unsigned hul = 0, hur = 0;
            if constexpr (BIG) {
                hul = T.wd[0][tid];
                hur = T.wd[1][tid];
            }
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const pkey_t k0 = B.k[r][c];
                    const unsigned hp = B.h[r][c];
                    const pkey_t u = r ? B.k[r - 1][c] : n[c + 1];
                    const pkey_t ul = r ? (c ? B.k[r - 1][c - 1] : w[r - 1]) : n[c];
                    const pkey_t ur = r ? (c < 3 ? B.k[r - 1][c + 1] : e[r - 1]) : n[c + 2];
                    const pkey_t l = c ? B.k[r][c - 1] : w[r];
                    const unsigned hu = r ? B.h[r - 1][c] : B.hn[c];
                    const unsigned hl = c ? B.h[r][c - 1] : B.hw[r];
                    const unsigned h_ul = r ? (c ? B.h[r - 1][c - 1] : B.hw[r - 1]) : c ? B.hn[c - 1] : hul;
                    const unsigned h_ur = r ? (c < 3 ? B.h[r - 1][c + 1] : B.he[r - 1]) : c < 3 ? B.hn[c + 1] : hur;
                    pkey_t k = kmin(k0, key_axis(u, hp, hu));
                    k = kmin(k, diag(ul, e_ul(r, c), hp, h_ul));
                    k = kmin(k, diag(ur, e_ur(r, c), hp, h_ur));
                    k = kmin(k, key_axis(l, hp, hl));
                    if (!FULL_TILE && !((B.valid >> (4 * r + c)) & 1u)) k = k0;
                    if (k != k0) now |= 1u << (4 * r + c);
                    B.k[r][c] = k;
                }
        }
        {
            pkey_t s[6];
#pragma unroll
            for (int c = 0; c < 6; ++c) s[c] = around(T.K, b, 4, c - 1);
            unsigned hll = 0, hlr = 0;
            if constexpr (BIG) {
                hll = T.wd[2][tid];
                hlr = T.wd[3][tid];
            }
#pragma unroll
            for (int r = 3; r >= 0; --r)
#pragma unroll
                for (int c = 3; c >= 0; --c) {
                    const pkey_t k0 = B.k[r][c];
                    const unsigned hp = B.h[r][c];
                    const pkey_t d = r < 3 ? B.k[r + 1][c] : s[c + 1];
                    const pkey_t dl = r < 3 ? (c ? B.k[r + 1][c - 1] : w[r + 1]) : s[c];
                    const pkey_t dr = r < 3 ? (c < 3 ? B.k[r + 1][c + 1] : e[r + 1]) : s[c + 2];
                    const pkey_t q = c < 3 ? B.k[r][c + 1] : e[r];
                    const unsigned hd = r < 3 ? B.h[r + 1][c] : B.hs[c];
                    const unsigned hq = c < 3 ? B.h[r][c + 1] : B.he[r];
                    const unsigned h_dl = r < 3 ? (c ? B.h[r + 1][c - 1] : B.hw[r + 1]) : c ? B.hs[c - 1] : hll;
                    const unsigned h_dr = r < 3 ? (c < 3 ? B.h[r + 1][c + 1] : B.he[r + 1]) : c < 3 ? B.hs[c + 1] : hlr;
                    pkey_t k = kmin(k0, key_axis(d, hp, hd));
                    k = kmin(k, diag(dl, e_ll(r, c), hp, h_dl));
                    k = kmin(k, diag(dr, e_lr(r, c), hp, h_dr));
                    k = kmin(k, key_axis(q, hp, hq));
                    if (!FULL_TILE && !((B.valid >> (4 * r + c)) & 1u)) k = k0;
                    if (k != k0) now |= 1u << (4 * r + c);
                    B.k[r][c] = k;
                }
        }
        if (now) {
            changed |= now;
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    if (r == 0 || r == 3 || c == 0 || c == 3) T.K[plane_of(r, c)][b] = B.k[r][c];
        }
        // each round that changes a key settles another block of some
        // shortest path, and a path in the tile has fewer blocks than pixels
        if (!__syncthreads_or(now != 0)) break;
        if (round >= cap) {
            if (tid == 0) set_status(st, EPIC_ERR_NOT_CONVERGED);
            break;
        }
    }
    return changed;
}

// The rarer forms (tiles cut by the image's right or lower edge, costs above
// 1.41 units), out of line so that their registers do not weigh on the main
// one.
template <int MAXR, bool BIG>
__device__ __noinline__ unsigned rounds_apart(SettleTile<MAXR> &T, Block *B, int b, int cap,
                                              RunState *st) {
    return rounds<MAXR, false, BIG>(T, *B, b, cap, st);
}

// Stage tile `g`: this thread's block into B, the tile's border keys and
// half-costs and the ring into shared memory; every thread has passed a
// barrier when it returns.  Cells outside the image are unreached with
// half-cost zero.  Row rv of the tile (the ring row below) may lie inside a
// block when the tile is not a whole number of blocks high; it is held like
// the ring, never updated.
template <int MAXR, typename Map = FrameMap>
__device__ void stage_tile(const PairDev &P, SettleTile<MAXR> &T, const TileGeo &g, Block &B,
                           RunState *st, const Map &map) {
    constexpr int NT = Dim<MAXR>::NT, NB = Dim<MAXR>::NB;
    const int tid = threadIdx.x, bx = tid & 15, by = tid >> 4;
    const int b = (by + 1) * RT_BX + bx + 1;
    const int W = P.W, H = P.H;
    const float *gc = P.C;
    const int nrow = min(4, min(g.rv + 1, H - g.y0) - 4 * by);
    const int ncol = min(4, g.wv - 4 * bx);
    B.valid = 0;
    float cc[4][4];
    const bool cvec = (W & 3) == 0 && ((uintptr_t)gc & 15) == 0;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const size_t o = (size_t)(g.y0 + 4 * by + r) * W + g.x0 + 4 * bx;
        const int nc = r < nrow ? ncol : 0;
        load_costs(gc, o, nc, cvec, cc[r]);
        map.row(g.x0 + 4 * bx, g.y0 + 4 * by + r, nc, B.k[r]);
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (c < nc && 4 * by + r < g.rv) B.valid |= 1u << (4 * r + c);
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
        rk[j] = KEY_INF;
        rc[j] = 0.f;
        if (in) {
            const size_t o = (size_t)gy * W + gx;
            rc[j] = __ldg(gc + o);
            rk[j] = map.at(gx, gy);
        }
    }
    HalfCost half(P);
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            B.h[r][c] = half(cc[r][c]);
            if (r == 0 || r == 3 || c == 0 || c == 3) {
                T.h[plane_of(r, c)][b] = B.h[r][c];
                T.K[plane_of(r, c)][b] = B.k[r][c];
            }
        }
#pragma unroll
    for (int j = 0; j < PER; ++j)
        if (re[j] >= 0) {
            (&T.h[0][0])[re[j]] = half(rc[j]);
            (&T.K[0][0])[re[j]] = rk[j];
        }
    if (half.bad) set_status(st, EPIC_ERR_INVALID);
    const unsigned hm = __reduce_max_sync(FULL, half.largest);
    if ((tid & 31) == 0) T.hmax[tid >> 5] = hm;
    if (tid == 0) T.flags = 0;
    __syncthreads();
}

// Solve the staged tile.  Reads the half-costs around the block, replaces the
// half-cost planes by the diagonal weights and runs the rounds.
template <int MAXR>
__device__ unsigned solve_tile(SettleTile<MAXR> &T, const TileGeo &g, Block &B, RunState *st) {
    constexpr int NW = Dim<MAXR>::NT / 32;
    const int tid = threadIdx.x, bx = tid & 15, by = tid >> 4;
    const int b = (by + 1) * RT_BX + bx + 1;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        B.hn[i] = around(T.h, b, -1, i);
        B.hs[i] = around(T.h, b, 4, i);
        B.hw[i] = around(T.h, b, i, -1);
        B.he[i] = around(T.h, b, i, 4);
    }
    const unsigned hul = around(T.h, b, -1, -1), hur = around(T.h, b, -1, 4);
    const unsigned hll = around(T.h, b, 4, -1), hlr = around(T.h, b, 4, 4);
    unsigned hm = T.hmax[0];
#pragma unroll
    for (int w = 1; w < NW; ++w) hm = max(hm, T.hmax[w]);
    __syncthreads();   // the planes are read; the weights take their place
    // sqrt(2) (h_p + h_q) fits 32 bits up to 2 h = 2^32 / sqrt(2)
    const bool big = hm > 1518500249u;
    if (tid == 0) T.big = big;
    if (!big) {
        auto put = [&](int e, unsigned hp, unsigned hq) { T.wd[e][tid] = (unsigned)step_diag(hp, hq); };
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const unsigned hp = B.h[r][c];
                put(e_ul(r, c), hp, r ? (c ? B.h[r - 1][c - 1] : B.hw[r - 1]) : c ? B.hn[c - 1] : hul);
                put(e_ur(r, c), hp, r ? (c < 3 ? B.h[r - 1][c + 1] : B.he[r - 1]) : c < 3 ? B.hn[c + 1] : hur);
                if (r == 3 || c == 0)
                    put(e_ll(r, c), hp, r < 3 ? B.hw[r + 1] : c ? B.hs[c - 1] : hll);
                if (r == 3 || c == 3)
                    put(e_lr(r, c), hp, r < 3 ? B.he[r + 1] : c < 3 ? B.hs[c + 1] : hlr);
            }
    } else {
        T.wd[0][tid] = hul;
        T.wd[1][tid] = hur;
        T.wd[2][tid] = hll;
        T.wd[3][tid] = hlr;
    }
    // (a thread reads only its own weights: no barrier)
    const int cap = 2 + RT_COLS * g.rv;
    if (big || g.wv < RT_COLS || g.rv < MAXR) {
        Block C = B;   // (B itself stays in registers)
        const unsigned changed = big ? rounds_apart<MAXR, true>(T, &C, b, cap, st)
                                     : rounds_apart<MAXR, false>(T, &C, b, cap, st);
#pragma unroll
        for (int i = 0; i < 16; ++i) B.k[i >> 2][i & 3] = C.k[i >> 2][i & 3];
        return changed;
    }
    return rounds<MAXR, true, false>(T, B, b, cap, st);
}

// Write the cells `mask` of this thread's block back to the key map.
__device__ __forceinline__ void write_block(const PairDev &P, const TileGeo &g, const Block &B,
                                            unsigned mask) {
    const int bx = threadIdx.x & 15, by = threadIdx.x >> 4;
    const bool kvec = (P.W & 1) == 0;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const unsigned m = (mask >> (4 * r)) & 15u;
        if (!m) continue;
        pkey_t *dst = P.keys + (size_t)(g.y0 + 4 * by + r) * P.W + g.x0 + 4 * bx;
        if (kvec && ((B.valid >> (4 * r)) & 15u) == 15u) {
            reinterpret_cast<ulonglong2 *>(dst)[0] = make_ulonglong2(B.k[r][0], B.k[r][1]);
            reinterpret_cast<ulonglong2 *>(dst)[1] = make_ulonglong2(B.k[r][2], B.k[r][3]);
        } else {
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if ((m >> c) & 1u) dst[c] = B.k[r][c];
        }
    }
}

// Which neighbours' border pixels, as the tile knows them, this thread's border
// pixels improve (TB_* bits; where weights need more than 32 bits, or the ring
// row lies among the blocks: by its changed border pixels alone).
template <int MAXR>
__device__ unsigned settle_offers(const SettleTile<MAXR> &T, const TileGeo &g, const Block &B,
                                  unsigned mask) {
    const int tid = threadIdx.x, bx = tid & 15, by = tid >> 4;
    const int b = (by + 1) * RT_BX + bx + 1;
    const bool big = T.big != 0;
    const int last = g.rv - 1 - 4 * by;   // the tile's bottom row in this block
    bool up = false, down = false, left = false, right = false;
    bool ul = false, ur = false, dl = false, dr = false;
    if (big || g.rv < MAXR) {
        up = by == 0 && (mask & 0xFu);
        down = last >= 0 && last < 4 && ((mask >> (4 * last)) & 0xFu);
        left = bx == 0 && (mask & 0x1111u);
        right = bx == 15 && (mask & 0x8888u);
        ul = up && left;
        ur = up && right;
        dl = down && left;
        dr = down && right;
    } else {
        auto axis = [&](int r, int c, int r2, int c2, unsigned h) {
            return key_axis(B.k[r][c], B.h[r][c], h) < around(T.K, b, r2, c2);
        };
        auto diag = [&](int r, int c, int r2, int c2, int e) {
            return key_plus(B.k[r][c], T.wd[e][tid]) < around(T.K, b, r2, c2);
        };
        if (by == 0) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                up |= axis(0, c, -1, c, B.hn[c]);
                if (c || bx) up |= diag(0, c, -1, c - 1, e_ul(0, c));
                if (c < 3 || bx < 15) up |= diag(0, c, -1, c + 1, e_ur(0, c));
            }
            ul = bx == 0 && diag(0, 0, -1, -1, e_ul(0, 0));
            ur = bx == 15 && diag(0, 3, -1, 4, e_ur(0, 3));
        }
        if (4 * by + 4 == MAXR) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                down |= axis(3, c, 4, c, B.hs[c]);
                if (c || bx) down |= diag(3, c, 4, c - 1, e_ll(3, c));
                if (c < 3 || bx < 15) down |= diag(3, c, 4, c + 1, e_lr(3, c));
            }
            dl = bx == 0 && diag(3, 0, 4, -1, e_ll(3, 0));
            dr = bx == 15 && diag(3, 3, 4, 4, e_lr(3, 3));
        }
        if (bx == 0) {
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                left |= axis(r, 0, r, -1, B.hw[r]);
                if (r || by) left |= diag(r, 0, r - 1, -1, e_ul(r, 0));
                if (4 * by + r + 1 < MAXR) left |= diag(r, 0, r + 1, -1, e_ll(r, 0));
            }
        }
        if (bx == 15) {
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                right |= axis(r, 3, r, 4, B.he[r]);
                if (r || by) right |= diag(r, 3, r - 1, 4, e_ur(r, 3));
                if (4 * by + r + 1 < MAXR) right |= diag(r, 3, r + 1, 4, e_lr(r, 3));
            }
        }
    }
    return (up ? TB_U : 0) | (down ? TB_D : 0) | (left ? TB_L : 0) | (right ? TB_R : 0) |
           (ul ? TB_UL : 0) | (ur ? TB_UR : 0) | (dl ? TB_DL : 0) | (dr ? TB_DR : 0);
}

// Settle tile (tx, ty): relax it to its fixed point with the ring around it.
// Returns what the solve did (TB_*; 0: nothing changed), the same in every
// thread; the changed keys are written back (own_tiles fences them).
template <int MAXR>
__device__ unsigned settle_tile(const PairDev &P, int tx, int ty, SettleTile<MAXR> &T, RunState *st) {
    const int tid = threadIdx.x;
    const TileGeo g = tile_geo(P, tx, ty);
    Block B;
    stage_tile(P, T, g, B, st, FrameMap(P));
    const unsigned mask = solve_tile(T, g, B, st);
    unsigned f = 0;
    if (mask) {
        write_block(P, g, B, mask);
        f = TB_ANY;
    }
    if (__syncthreads_or(mask != 0)) f |= settle_offers(T, g, B, mask);
    f = __reduce_or_sync(FULL, f);
    if (f && (tid & 31) == 0) atomicOr(&T.flags, f);
    __syncthreads();
    return T.flags;
}

}  // namespace

}  // namespace epic
