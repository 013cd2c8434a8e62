// Exact variant (Sec. 5.2, Table 2): every pixel takes its own K nearest
// matches under the exact distance and its own fit, instead of inheriting
// the model of its Voronoi cell (the approximation of Eq. 4).
//
//   bin_kernel         Euclidean: the matches by cells of the frame;
//   weight_kernel      Euclidean: kernel weights by squared distance (pixel
//                      centres are integers, so few distances differ);
//   fit_kernel         a CTA takes 8 x 8 pixels, a thread each.  The
//                      candidates that any of them can need are gathered
//                      (Euclidean: all matches within the K-th distance of
//                      the group's centre plus twice its radius; geodesic:
//                      the matches whose single-source distances reach the
//                      group, from k_single.cu), sorted once by their
//                      distance from the centre, and each thread keeps its K
//                      smallest keys (distance, index) by insertion: in an
//                      order that is nearly its own, an insertion moves few
//                      entries.  Then it fits Eq. 2 centred at the pixel (FP64
//                      sums and solve; the NW estimate of Eq. 1 when
//                      degenerate or requested) and writes the model's value
//                      at the pixel.
//   scan_kernel        groups with more candidates than fit in shared memory
//                      (dense clusters), or all groups (scan_all): every
//                      candidate in index order, into 64-bit keys.
//
// 1024 x 436 pixels, 5000 matches, K = 100: 1.83 ms (Euclidean) and 4.9 + 1.3
// ms (geodesic; the second for the groups left to scan_kernel), against 28.0
// and 13.9 ms for one scan of all 5000 candidates per pixel.  What bounds it: the FP64 pipe (2 fused multiply-adds per SM and
// cycle; 16 per neighbour and pixel with tabulated weights, ~36 with an
// exponential each).
#include "epic_internal.cuh"

namespace epic {

namespace {

constexpr int GROUP = 8;               // a CTA's pixels: GROUP x GROUP
constexpr float GROUP_RADIUS = 5.66f;  // farthest pixel from its centre pixel
constexpr int CAND_BITS = 9;
constexpr int CAND = 1 << CAND_BITS;   // candidates of a group in shared memory
static_assert(LABEL_BITS + CAND_BITS <= 32, "a match and a place in a word");
constexpr int BIN_CELLS = 8192;
constexpr int BIN_THREADS = 1024;
constexpr float FAR = 2040.f;          // beyond: squared distances leave a packed key
static_assert(EXACT_THREADS == GROUP * GROUP, "a thread a pixel");

__device__ __forceinline__ float inf() { return __int_as_float(0x7f800000); }

// Squared distance between a pixel and a match's source pixel, and the
// distance as the fit takes it.
__device__ __forceinline__ float dist2(float px, float py, float mx, float my) {
    const float dx = __fsub_rn(px, mx), dy = __fsub_rn(py, my);
    return __fmaf_rn(dx, dx, __fmul_rn(dy, dy));
}
__device__ __forceinline__ float source(float x) { return floorf(x + 0.5f); }

// One CTA: matches by cells of 2^shift x 2^shift pixels (those outside the
// image in the cell nearest to them; those without a finite position, which no
// pixel is at a finite distance from, in none).
__global__ void __launch_bounds__(BIN_THREADS) bin_kernel(const float4 *matches, int N, int W, int H,
                                                          int shift, int cells_x, int cells,
                                                          int *cell_start, int *cell_match) {
    __shared__ int count[BIN_CELLS];
    __shared__ int warp_sums[32];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    for (int i = tid; i < BIN_CELLS; i += BIN_THREADS) count[i] = 0;
    __syncthreads();
    auto cell = [&](int m) {
        const float4 q = __ldg(matches + m);
        const float x = source(q.x), y = source(q.y);
        if (!isfinite(x) || !isfinite(y)) return -1;
        const int cx = (int)fminf(fmaxf(x, 0.f), (float)(W - 1)) >> shift;
        const int cy = (int)fminf(fmaxf(y, 0.f), (float)(H - 1)) >> shift;
        return cy * cells_x + cx;
    };
    for (int m = tid; m < N; m += BIN_THREADS) {
        const int c = cell(m);
        if (c >= 0) atomicAdd(&count[c], 1);
    }
    __syncthreads();
    constexpr int PER = BIN_CELLS / BIN_THREADS;
    int x[PER], sum = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        x[j] = count[tid * PER + j];
        sum += x[j];
    }
    int sc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, sc, o);
        if (lane >= o) sc += t;
    }
    if (lane == 31) warp_sums[wid] = sc;
    __syncthreads();
    if (wid == 0) {
        int ws = warp_sums[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, ws, o);
            if (lane >= o) ws += t;
        }
        warp_sums[lane] = ws;
    }
    __syncthreads();
    int at = sc - sum + (wid ? warp_sums[wid - 1] : 0);
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int c = tid * PER + j;
        count[c] = at;   // the fill cursor
        if (c <= cells) cell_start[c] = at;
        at += x[j];
    }
    if (tid == BIN_THREADS - 1 && cells == BIN_CELLS) cell_start[cells] = at;
    __syncthreads();
    for (int m = tid; m < N; m += BIN_THREADS) {
        const int c = cell(m);
        if (c >= 0) cell_match[atomicAdd(&count[c], 1)] = m;
    }
}

__device__ __forceinline__ double kernel_weight(float a, float d) { return exp(-(double)a * (double)d); }

// Kernel weight of every squared distance below EXACT_WEIGHTS.
__global__ void weight_kernel(float a, double *table) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < EXACT_WEIGHTS) table[i] = kernel_weight(a, __fsqrt_rn((float)i));
}

// The weighted sums of Eq. 2 about a pixel, neighbours in key order.
struct Sums {
    double M00 = 0, M01 = 0, M02 = 0, M11 = 0, M12 = 0, M22 = 0;
    double ru0 = 0, ru1 = 0, ru2 = 0, rv0 = 0, rv1 = 0, rv2 = 0;
    __device__ __forceinline__ void add(double w, double xt, double yt, double u, double v) {
        M00 += w * xt * xt; M01 += w * xt * yt; M02 += w * xt;
        M11 += w * yt * yt; M12 += w * yt; M22 += w;
        ru0 += w * xt * u; ru1 += w * yt * u; ru2 += w * u;
        rv0 += w * xt * v; rv1 += w * yt * v; rv2 += w * v;
    }
    // The flow at the centre (the constant term of the fit), unless the fit
    // is degenerate.
    __device__ __forceinline__ bool solve(int cnt, float eps, float *fu, float *fv) const {
        const double c00 = M11 * M22 - M12 * M12;
        const double c01 = M12 * M02 - M01 * M22;
        const double c02 = M01 * M12 - M11 * M02;
        const double c12 = M01 * M02 - M00 * M12;
        const double c22 = M00 * M11 - M01 * M01;
        const double det = M00 * c00 + M01 * c01 + M02 * c02;
        const double tr3 = (M00 + M11 + M22) / 3.0;
        if (!(cnt >= 3 && det > (double)eps * tr3 * tr3 * tr3)) return false;
        const double id = 1.0 / det;
        *fu = (float)((c02 * ru0 + c12 * ru1 + c22 * ru2) * id);
        *fv = (float)((c02 * rv0 + c12 * rv1 + c22 * rv2) * id);
        return true;
    }
};

struct Cand {
    double x, y, u, v;   // a match's source position and flow
};
__device__ __forceinline__ Cand cand_of(float4 q) {
    return Cand{(double)q.x, (double)q.y, (double)q.z - (double)q.x, (double)q.w - (double)q.y};
}

// Shared memory of fit_kernel: the threads' sorted lists (entry j of thread t
// at j * EXACT_THREADS + t), then the candidates, first as they are selected,
// then as they are fitted.
struct Select {
    // distance from the centre << 32 | match (geodesic: match << 9 | place as
    // gathered): equal distances (frames of cost zero, matches on one pixel) come
    // in the order that the insertions below want (as gathered, which is any
    // order, 1024 x 436 of cost zero, 300 matches, K = 200: 59 ms; so: 21)
    unsigned long long key[CAND];
    float2 xy[CAND];                // Euclidean: source pixels, in key order; geodesic: the distance
                                    // tiles in y, as gathered
    int slot[CAND];                 // geodesic: distance tiles, in key order
    unsigned short id[CAND];        // rank of the match index among the candidates, in key order
};
union Work {
    Select s;
    Cand c[CAND];                   // by rank
};
__host__ __device__ __forceinline__ size_t list_bytes(int K, bool geo) {
    // (geodesic: distance and rank apart; Euclidean: squared distance << 9 | rank)
    return (size_t)K * EXACT_THREADS * (geo ? 6 : 4);
}
__host__ __device__ __forceinline__ size_t fit_smem_bytes(int K, bool geo) {
    return ((list_bytes(K, geo) + 15) & ~(size_t)15) + sizeof(Work) + CAND * sizeof(int);
}

// Ascending bitonic sort of n keys (padded with ~0 to a power of two) by the
// CTA.
__device__ void sort_keys(unsigned long long *key, int n) {
    int size = 2;
    while (size < n) size <<= 1;
    for (int i = n + threadIdx.x; i < size; i += EXACT_THREADS) key[i] = ~0ull;
    __syncthreads();
    for (int k = 2; k <= size; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = threadIdx.x; i < size / 2; i += EXACT_THREADS) {
                const int a = 2 * i - (i & (j - 1)), b = a + j;
                const bool up = (a & k) == 0;
                const unsigned long long x = key[a], y = key[b];
                if ((x > y) == up) {
                    key[a] = y;
                    key[b] = x;
                }
            }
            __syncthreads();
        }
}

// Euclidean: the radius around a group's centre in which candidates are first
// looked for: the K-th distance at the mean density, and some.
__host__ __device__ __forceinline__ float first_radius(const ExactArgs &x) {
    return 1.25f * sqrtf((float)x.K * (float)x.W * (float)x.H / (3.1416f * (float)x.N)) + 2.f * GROUP_RADIUS + 4.f;
}
// Whether all groups are scanned: so few matches that gathering and sorting them
// costs more (1024 x 436: one match 105 us scanned and 138 by groups, 33 of K = 10
// 451 and 488, 48 of K = 10 449 and 452, 64 of K = 64 2.5 and 3.1 ms, 100 of K =
// 100 4.7 and 4.6 ms), or so many that at the mean density a group needs more
// than shared memory holds (128 x 128, a match per pixel, K = 32: 4.5 ms, and 4.6
// with the look at the groups before it).
constexpr int SCAN_FEW = 24, SCAN_MOST = 80;
bool scan_all(const ExactArgs &x) {
    if (x.N <= SCAN_MOST && x.N <= SCAN_FEW + x.K) return true;
    const float per = (float)x.N / ((float)x.W * (float)x.H);
    const float need = sqrtf((float)x.K / (3.1416f * per)) + 2.f * GROUP_RADIUS;
    return x.N > CAND && 3.1416f * need * need * per > 1.1f * (float)CAND;
}

template <bool GEO>
__global__ void __launch_bounds__(EXACT_THREADS) fit_kernel(ExactArgs x, int groups_x) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int t = threadIdx.x, lane = t & 31;
    const int K = x.K, W = x.W, H = x.H;
    float *ld = reinterpret_cast<float *>(smem);                                   // geodesic
    unsigned short *li = reinterpret_cast<unsigned short *>(ld + (size_t)K * EXACT_THREADS);
    unsigned *lk = reinterpret_cast<unsigned *>(smem);                             // Euclidean
    Work &w = *reinterpret_cast<Work *>(smem + ((list_bytes(K, GEO) + 15) & ~(size_t)15));
    int *match = reinterpret_cast<int *>(&w + 1);                                  // by rank
    __shared__ int s_n;
    // a group's pixels: warp 0 the upper 8 x 4, warp 1 the lower
    const int gx = (int)(blockIdx.x % groups_x) * GROUP, gy = (int)(blockIdx.x / groups_x) * GROUP;
    const int px = gx + (t & 7), py = gy + (t >> 3);
    const bool in = px < W && py < H;
    const int cx = min(gx + GROUP / 2, W - 1), cy = min(gy + GROUP / 2, H - 1);   // the centre
    const float fpx = (float)px, fpy = (float)py;
    int n = 0;
    bool fits = true;

    // ---- candidates, by their distance from the centre
    if constexpr (!GEO) {
        const float all = (float)(W + H);   // from here on every cell is looked at
        float S = fminf(all, first_radius(x));
        bool narrowed = false;
        for (int round = 0; round < 64; ++round) {
            if (t == 0) s_n = 0;
            __syncthreads();
            const bool every = S >= all;
            const int c0 = max(0, (int)((float)cx - S)) >> x.cell_shift;
            const int c1 = (int)fminf((float)cx + S, (float)(W - 1)) >> x.cell_shift;
            const int r0 = max(0, (int)((float)cy - S)) >> x.cell_shift;
            const int r1 = (int)fminf((float)cy + S, (float)(H - 1)) >> x.cell_shift;
            for (int r = r0; r <= r1; ++r) {
                // the cells of a row are consecutive
                const int i0 = __ldg(x.cell_start + r * x.cells_x + c0);
                const int i1 = __ldg(x.cell_start + r * x.cells_x + c1 + 1);
                for (int i = i0 + t; i < i1; i += EXACT_THREADS) {
                    const int m = __ldg(x.cell_match + i);
                    const float4 q = __ldg(x.matches + m);
                    const float d = __fsqrt_rn(dist2((float)cx, (float)cy, source(q.x), source(q.y)));
                    if (every ? d < inf() : d <= S) {
                        const int at = atomicAdd(&s_n, 1);
                        if (at < CAND)
                            w.s.key[at] = ((unsigned long long)__float_as_uint(d) << 32) | (unsigned)m;
                    }
                }
            }
            __syncthreads();
            n = s_n;
            __syncthreads();
            if (n > CAND) {
                // the first look may take in more than is needed: once, look
                // at a part of it (1024 x 436, a match for four pixels, K =
                // 100: 3.8 ms; 326 ms when such groups were left to the scan)
                if (narrowed) {
                    fits = false;
                    break;
                }
                narrowed = true;
                S *= sqrtf(0.9f * (float)CAND / (float)n);
                continue;
            }
            if (n < K && !every) {   // (K <= N; fewer may be at a finite distance)
                S = fminf(all, 1.5f * S);
                continue;
            }
            sort_keys(w.s.key, n);
            if (every) break;
            // every pixel of the group has K matches within R + radius, and
            // those within that of it are within R + 2 radius of the centre
            const float R = __uint_as_float((unsigned)(w.s.key[K - 1] >> 32)) + 2.f * GROUP_RADIUS + 0.1f;
            if (R <= S) {
                if (t == 0) s_n = 0;
                __syncthreads();
                int c = 0;
                for (int i = t; i < n; i += EXACT_THREADS)
                    c += __uint_as_float((unsigned)(w.s.key[i] >> 32)) <= R;
                c = __reduce_add_sync(0xffffffffu, c);
                if (lane == 0) atomicAdd(&s_n, c);
                __syncthreads();
                n = s_n;
                break;
            }
            S = fminf(all, R + 0.5f);
            __syncthreads();
        }
        // packed keys hold squared distances up to 2^22
        if (fits && n > 0 && !(__uint_as_float((unsigned)(w.s.key[n - 1] >> 32)) < FAR)) fits = false;
    } else {
        // the matches of the solve tile that reach a pixel of the group
        const int tile = (gy / 32) * x.tiles_x + gx / 64;
        const int e0 = __ldg(x.tile_start + tile), e1 = __ldg(x.tile_start + tile + 1);
        const int coff = (cy & 31) * 64 + (cx & 63);
        if (t == 0) s_n = 0;
        __syncthreads();
        // a warp takes 32 entries at a time: which of them reach one of all 64
        // pixels, and their distances at the centre
        for (int b = e0 + (t & 32); b < e1; b += EXACT_THREADS) {
            const int e = b + lane;
            const int2 ent = e < e1 ? __ldg(x.tile_entry + e) : make_int2(0, -1);
            unsigned reach = 0;
            for (int j = 0; j < 32 && b + j < e1; ++j) {
                const float *s = x.slots + (size_t)__shfl_sync(0xffffffffu, ent.y, j) * SINGLE_TILE;
                // lane: two pixels of the group
                const int q = 2 * lane;
                const int qx = gx + (q & 7), qy = gy + (q >> 3);
                const int o = (qy & 31) * 64 + (qx & 63);
                bool r = false;
                if (qy < H) r = (qx < W && __ldg(s + o) < inf()) || (qx + 1 < W && __ldg(s + o + 1) < inf());
                if (__any_sync(0xffffffffu, r)) reach |= 1u << j;
            }
            if ((reach >> lane) & 1u) {
                const int at = atomicAdd(&s_n, 1);
                if (at < CAND) {
                    const float d = __ldg(x.slots + (size_t)ent.y * SINGLE_TILE + coff);
                    w.s.key[at] = ((unsigned long long)__float_as_uint(d) << 32) |
                                  ((unsigned)ent.x << CAND_BITS) | (unsigned)at;
                    w.s.xy[at].y = __int_as_float(ent.y);
                }
            }
        }
        __syncthreads();
        n = s_n;
        fits = n <= CAND;
        if (fits) sort_keys(w.s.key, n);
    }
    if (!fits) {
        if (t == 0) x.slow_list[atomicAdd(x.slow_count, 1)] = (int)blockIdx.x;
        return;
    }
    __syncthreads();
    // ---- ranks of the match indices (ties go to the smaller index)
    if constexpr (GEO) {
        for (int i = t; i < n; i += EXACT_THREADS)
            w.s.slot[i] = __float_as_int(w.s.xy[(unsigned)w.s.key[i] & (CAND - 1)].y);
    } else {
        for (int i = t; i < n; i += EXACT_THREADS) {
            const float4 q = __ldg(x.matches + (unsigned)w.s.key[i]);
            w.s.xy[i] = make_float2(source(q.x), source(q.y));
        }
    }
    __syncthreads();
    for (int i = t; i < n; i += EXACT_THREADS) {
        auto index = [&](int j) { return (int)((unsigned)w.s.key[j] >> (GEO ? CAND_BITS : 0)); };
        const int m = index(i);
        int r = 0;
        for (int j = 0; j < n; ++j) r += index(j) < m;
        w.s.id[i] = (unsigned short)r;
        match[r] = m;
    }
    __syncthreads();
    // ---- the K smallest keys, by insertion into the thread's sorted list
    int cnt = 0;
    if constexpr (GEO) {
        const int off = (py & 31) * 64 + (px & 63);
        for (int i0 = 0; i0 < n; i0 += 8) {
            float dg[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                dg[u] = in && i0 + u < n ? __ldg(x.slots + (size_t)w.s.slot[i0 + u] * SINGLE_TILE + off) : inf();
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const float d = dg[u];
                // (beyond the single-source run's cap: not among the K nearest)
                if (!(d < inf())) continue;
                const unsigned short id = w.s.id[i0 + u];
                auto less = [&](int j) {   // this key before entry j's?
                    const float dj = ld[j * EXACT_THREADS + t];
                    return d < dj || (d == dj && id < li[j * EXACT_THREADS + t]);
                };
                int j;
                if (cnt < K) j = cnt++;
                else if (less(K - 1)) j = K - 1;
                else continue;
                for (; j > 0 && less(j - 1); --j) {
                    ld[j * EXACT_THREADS + t] = ld[(j - 1) * EXACT_THREADS + t];
                    li[j * EXACT_THREADS + t] = li[(j - 1) * EXACT_THREADS + t];
                }
                ld[j * EXACT_THREADS + t] = d;
                li[j * EXACT_THREADS + t] = id;
            }
        }
    } else {
        unsigned last = 0;
        for (int i = 0; i < n; ++i) {
            const float2 m = w.s.xy[i];
            const unsigned key = ((unsigned)dist2(fpx, fpy, m.x, m.y) << 9) | w.s.id[i];
            int j;
            if (cnt < K) j = cnt++;
            else if (key < last) j = K - 1;
            else continue;
            for (; j > 0; --j) {
                const unsigned p = lk[(j - 1) * EXACT_THREADS + t];
                if (p < key) break;
                lk[j * EXACT_THREADS + t] = p;
            }
            lk[j * EXACT_THREADS + t] = key;
            if (cnt == K) last = lk[(K - 1) * EXACT_THREADS + t];
        }
    }
    __syncthreads();
    // ---- the fit
    for (int i = t; i < n; i += EXACT_THREADS) w.c[i] = cand_of(__ldg(x.matches + match[i]));
    __syncthreads();
    if (!in) return;
    const long long p = (long long)py * W + px;
    auto entry = [&](int j, int *id, float *d) -> double {   // and its kernel weight
        if constexpr (GEO) {
            *id = li[j * EXACT_THREADS + t];
            *d = ld[j * EXACT_THREADS + t];
            return kernel_weight(x.a, *d);
        } else {
            const unsigned key = lk[j * EXACT_THREADS + t];
            *id = (int)(key & (CAND - 1));
            *d = __fsqrt_rn((float)(key >> 9));
            return key >> 9 < EXACT_WEIGHTS ? __ldg(x.weights + (key >> 9)) : kernel_weight(x.a, *d);
        }
    };
    Sums s;
    if (x.estimator == 0)
        for (int j = 0; j < cnt; ++j) {
            int id;
            float d;
            const double k = entry(j, &id, &d);
            const Cand q = w.c[id];
            s.add(x.weight_squared ? k * k : k, q.x - px, q.y - py, q.u, q.v);
        }
    float fu, fv;
    if (x.estimator != 0 || !s.solve(cnt, x.fallback_eps, &fu, &fv)) {
        // the NW estimate
        double sk = 0, sku = 0, skv = 0;
        for (int j = 0; j < cnt; ++j) {
            int id;
            float d;
            const double k = entry(j, &id, &d);
            const Cand q = w.c[id];
            sk += k;
            sku += k * q.u;
            skv += k * q.v;
        }
        fu = (float)(sku / sk);
        fv = (float)(skv / sk);
    }
    x.flow[2 * p] = fu;
    x.flow[2 * p + 1] = fv;
    if (x.knn_idx)
        for (int j = 0; j < K; ++j) {
            int id = 0;
            float d = inf();
            if (j < cnt) entry(j, &id, &d);
            x.knn_idx[p * K + j] = j < cnt ? match[id] : -1;
            x.knn_dist[p * K + j] = d;
        }
}

// The groups that fit_kernel left, or all of them: every candidate in index
// order, a thread a pixel, sorted insertion of 64-bit keys (distance, index).
template <bool GEO>
__global__ void __launch_bounds__(EXACT_THREADS) scan_kernel(ExactArgs x, int groups_x, int all) {
    extern __shared__ __align__(16) unsigned char smem[];
    unsigned long long *list = reinterpret_cast<unsigned long long *>(smem);
    const int T = EXACT_THREADS, t = threadIdx.x, K = x.K;
    const int count = all ? all : *(volatile const int *)x.slow_count;
    for (int g = blockIdx.x; g < count; g += gridDim.x) {
        const int grp = all ? g : x.slow_list[g];
        const int gx = grp % groups_x * GROUP, gy = grp / groups_x * GROUP;
        const int px = gx + (t & 7), py = gy + (t >> 3);
        if (px >= x.W || py >= x.H) continue;
        const int tile = GEO ? (gy / 32) * x.tiles_x + gx / 64 : 0;
        const int e0 = GEO ? x.tile_start[tile] : 0, e1 = GEO ? x.tile_start[tile + 1] : x.N;
        int cnt = 0;
        // (SCAN distances at a time, for their loads to overlap)
        constexpr int SCAN = 8;
        for (int b = e0; b < e1; b += SCAN) {
            float dg[SCAN];
            int mg[SCAN];
#pragma unroll
            for (int u = 0; u < SCAN; ++u) {
                const int e = b + u;
                dg[u] = inf();
                mg[u] = e;
                if (e >= e1) continue;
                if (GEO) {
                    const int2 ent = __ldg(x.tile_entry + e);
                    mg[u] = ent.x;
                    dg[u] = __ldg(x.slots + (size_t)ent.y * SINGLE_TILE + (py & 31) * 64 + (px & 63));
                } else {
                    const float4 q = __ldg(x.matches + e);
                    dg[u] = __fsqrt_rn(dist2((float)px, (float)py, source(q.x), source(q.y)));
                }
            }
#pragma unroll
            for (int u = 0; u < SCAN; ++u) {
                const float d = dg[u];
                if (!(d < inf())) continue;
                const unsigned long long key = ((unsigned long long)__float_as_uint(d) << 32) | (unsigned)mg[u];
                int j;
                if (cnt < K) j = cnt++;
                else if (key < list[(K - 1) * T + t]) j = K - 1;
                else continue;
                for (; j > 0 && list[(j - 1) * T + t] > key; --j) list[j * T + t] = list[(j - 1) * T + t];
                list[j * T + t] = key;
            }
        }
        const long long p = (long long)py * x.W + px;
        Sums s;
        double sk = 0, sku = 0, skv = 0;
        for (int j = 0; j < K; ++j) {
            if (j >= cnt) {
                if (x.knn_idx) {
                    x.knn_idx[p * K + j] = -1;
                    x.knn_dist[p * K + j] = inf();
                }
                continue;
            }
            const unsigned long long key = list[j * T + t];
            const float d = __uint_as_float((unsigned)(key >> 32));
            const Cand q = cand_of(__ldg(x.matches + (unsigned)key));
            const double k = kernel_weight(x.a, d);
            s.add(x.weight_squared ? k * k : k, q.x - px, q.y - py, q.u, q.v);
            sk += k;
            sku += k * q.u;
            skv += k * q.v;
            if (x.knn_idx) {
                x.knn_idx[p * K + j] = (int)(unsigned)key;
                x.knn_dist[p * K + j] = d;
            }
        }
        float fu, fv;
        if (x.estimator != 0 || !s.solve(cnt, x.fallback_eps, &fu, &fv)) {
            fu = (float)(sku / sk);
            fv = (float)(skv / sk);
        }
        x.flow[2 * p] = fu;
        x.flow[2 * p + 1] = fv;
    }
}

// Seed offsets of the cap map (in key units): an upper bound of each
// match's K-th nearest graph distance, from the K-NN lists of an
// approximate run.  A graph distance is the cost of a real path (each edge
// weight is one), but summed in float from float-rounded weights, hence the
// relative and absolute margins.  Fewer than K neighbours: no bound.
__global__ void cap_seed_kernel(const float *knn_dist, const int *knn_count, int N, int K,
                                int ld, unsigned long long *init) {
    constexpr unsigned long long UNBOUNDED = 1ull << 40;
    for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < N; m += gridDim.x * blockDim.x) {
        unsigned long long u = UNBOUNDED;
        if (knn_count[m] >= K) {
            const double d = (double)knn_dist[(size_t)m * ld + K - 1];
            if (d >= 0.0 && d < 256.0)
                u = min((unsigned long long)ceil(d * 2147483648.0 * (1.0 + 1.0 / 65536.0)) + 256ull,
                        UNBOUNDED);
        }
        init[m] = u;
    }
}

template <bool GEO>
cudaError_t fit_launch(const ExactArgs &x, int num_sms, cudaStream_t stream) {
    const size_t smem = fit_smem_bytes(x.K, GEO), slow = exact_smem_bytes(x.K);
    cudaError_t e = cudaFuncSetAttribute(fit_kernel<GEO>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(scan_kernel<GEO>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)slow);
    if (e != cudaSuccess) return e;
    const int groups_x = (x.W + GROUP - 1) / GROUP;
    const long long groups = exact_groups(x.H, x.W);
    if (!GEO && scan_all(x)) {
        scan_kernel<GEO><<<(unsigned)groups, EXACT_THREADS, slow, stream>>>(x, groups_x, (int)groups);
        return cudaGetLastError();
    }
    if ((e = cudaMemsetAsync(x.slow_count, 0, sizeof(int), stream)) != cudaSuccess) return e;
    fit_kernel<GEO><<<(unsigned)groups, EXACT_THREADS, smem, stream>>>(x, groups_x);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int blocks = (int)(groups < 4LL * num_sms ? groups : 4LL * num_sms);
    scan_kernel<GEO><<<blocks, EXACT_THREADS, slow, stream>>>(x, groups_x, 0);
    return cudaGetLastError();
}

}  // namespace

size_t exact_smem_bytes(int K) { return (size_t)K * EXACT_THREADS * sizeof(unsigned long long); }

long long exact_groups(int H, int W) {
    return (long long)((W + GROUP - 1) / GROUP) * ((H + GROUP - 1) / GROUP);
}

void exact_cells(int H, int W, int *shift, int *cells_x, int *cells) {
    for (int s = 4;; ++s) {
        const long long cx = ((long long)W + (1 << s) - 1) >> s, cy = ((long long)H + (1 << s) - 1) >> s;
        if (cx * cy > BIN_CELLS) continue;
        *shift = s;
        *cells_x = (int)cx;
        *cells = (int)(cx * cy);
        return;
    }
}

cudaError_t launch_cap_seed(const float *knn_dist, const int *knn_count, int N, int K, int ld,
                            unsigned long long *init, cudaStream_t stream) {
    const int blocks = (N + 255) / 256 < 1024 ? (N + 255) / 256 : 1024;
    cap_seed_kernel<<<blocks < 1 ? 1 : blocks, 256, 0, stream>>>(knn_dist, knn_count, N, K, ld, init);
    return cudaGetLastError();
}

cudaError_t launch_exact_euclidean(const ExactArgs &x, int *cell_start, int *cell_match, double *weights,
                                   int cells, int num_sms, cudaStream_t stream) {
    if (!scan_all(x)) {
        bin_kernel<<<1, BIN_THREADS, 0, stream>>>(x.matches, x.N, x.W, x.H, x.cell_shift, x.cells_x, cells,
                                                  cell_start, cell_match);
        weight_kernel<<<(EXACT_WEIGHTS + 255) / 256, 256, 0, stream>>>(x.a, weights);
    }
    const cudaError_t e = cudaGetLastError();
    return e ? e : fit_launch<false>(x, num_sms, stream);
}

cudaError_t launch_exact_geodesic(const ExactArgs &x, int num_sms, cudaStream_t stream) {
    return fit_launch<true>(x, num_sms, stream);
}

}  // namespace epic
