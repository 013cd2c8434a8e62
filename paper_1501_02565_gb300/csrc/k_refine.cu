// Variational refinement (Sec. 4, "Variational Energy Minimization"): the
// interpolated flow is refined at full resolution by fixed-point iterations,
// each linearising the data term (colour and gradient constancy with
// normalisation) at the current flow and solving the linear system of the
// Euler-Lagrange equations for the update with red-black SOR.
//
// Per fixed-point iteration:
//   coefficients   I2 is warped by the flow (in shared memory, with the pixels
//                  around a tile); per pixel the 2x2 data matrix A,
//                  right-hand side b (with the robust weights taken at zero
//                  update) and the smoothness weight
//                  phi = alpha Psi'(|grad u|^2 + |grad v|^2);
//   SOR            half-sweeps (colours alternating), then w += (du, dv).
// Frames whose pixels fit on the chip in one wave of CTAs (up to 450 to 500
// K pixels, by their shape) run in one cooperative launch of sor_kernel; larger
// ones launch coeff_kernel, sor_kernel per SOR_H half-sweeps, update_kernel.
// Derivatives are central differences on the edge-replicated image, nested
// the same way for second derivatives (the derivative image is itself
// edge-replicated).  All arithmetic is float32.
#include <algorithm>
#include <type_traits>

#include "epic_internal.cuh"
#include "quotient.cuh"

namespace epic {

namespace {

constexpr int SOR_H = 6;            // half-sweeps between exchanges (even: each begins with red)
constexpr int SOR_MAX_TILES = 1024;
static_assert(SOR_H % 2 == 0, "a round begins with red");

// Scratch of a refinement: coefficients by pixel, split as sor_kernel reads
// them; two update buffers; sor_kernel's progress by tile and its error word.
struct RefineScratch {
    float4 *a;      // [P] A11, A12, A22, b1
    float2 *b;      // [P] b2, phi
    union {
        float2 *d[2];           // [P] updates (frames of several waves)
        ulonglong2 *swap[2];    // [P] tagged updates of the cells near the cores' edges
    };
    unsigned *progress;
};

// Coefficients of the w x h pixels from (X0, Y0), by the CTA.  s: both images
// with two pixels around, channel by channel, 2 C (w + 4) (h + 4) words.  What
// other CTAs of the launch write (the flow) is read through L2.
template <int C>
__device__ void coeff_tile(const float *__restrict__ I1, const float *__restrict__ I2, const float2 *flow, int W,
                           int H, const RefineArgs &r, const RefineScratch &o, int X0, int Y0, int w, int h,
                           float *s) {
    const int tid = threadIdx.x, NT = blockDim.x, rw = w + 4, n = rw * (h + 4);
    X0 -= 2;
    Y0 -= 2;
    // I1, and I2 warped by the flow: I2w(p) = I2(p + w(p)), bilinear,
    // coordinates clamped
    for (int i = tid; i < n; i += NT) {
        const int ry = i / rw, x = X0 + i - ry * rw, y = Y0 + ry;
        if (x < 0 || x >= W || y < 0 || y >= H) continue;
        const size_t p = (size_t)y * W + x;
        const float2 f = __ldcg(flow + p);
        const float X = fminf(fmaxf((float)x + f.x, 0.f), (float)(W - 1));
        const float Y = fminf(fmaxf((float)y + f.y, 0.f), (float)(H - 1));
        const int xa = W > 1 ? min((int)floorf(X), W - 2) : 0;
        const int ya = H > 1 ? min((int)floorf(Y), H - 2) : 0;
        const int xb = min(xa + 1, W - 1), yb = min(ya + 1, H - 1);
        const float ax = X - (float)xa, ay = Y - (float)ya;
        // (which products are fused is written out: the compiler chooses by C)
        const float bx = __fsub_rn(1.f, ax), by = __fsub_rn(1.f, ay);
        const float *r0 = I2 + (size_t)ya * W * C, *r1 = I2 + (size_t)yb * W * C;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            s[c * n + i] = __ldg(I1 + p * C + c);
            const float a00 = __ldg(r0 + xa * C + c);
            const float a01 = __ldg(r0 + xb * C + c);
            const float a10 = __ldg(r1 + xa * C + c);
            const float a11 = __ldg(r1 + xb * C + c);
            s[(C + c) * n + i] = __fmaf_rn(by, __fmaf_rn(bx, a00, __fmul_rn(ax, a01)),
                                           __fmul_rn(ay, __fmaf_rn(bx, a10, __fmul_rn(ax, a11))));
        }
    }
    __syncthreads();
    for (int i = tid; i < w * h; i += NT) {
        const int ry = i / w, x = X0 + 2 + i - ry * w, y = Y0 + 2 + ry;
        if (x >= W || y >= H) continue;
        const size_t p = (size_t)y * W + x;
        // neighbours, and the neighbours' neighbours (the derivative images are
        // edge-replicated themselves)
        const int xl = max(x - 1, 0), xr = min(x + 1, W - 1), yu = max(y - 1, 0), yd = min(y + 1, H - 1);
        const int xll = max(xl - 1, 0) - X0, xlr = min(xl + 1, W - 1) - X0;
        const int xrl = max(xr - 1, 0) - X0, xrr = min(xr + 1, W - 1) - X0;
        const int yuu = max(yu - 1, 0) - Y0, yud = min(yu + 1, H - 1) - Y0;
        const int ydu = max(yd - 1, 0) - Y0, ydd = min(yd + 1, H - 1) - Y0;
        const int jx = x - X0, jl = xl - X0, jr = xr - X0, jy = y - Y0, ju = yu - Y0, jd = yd - Y0;
        auto at = [&](const float *s, int cx, int cy) { return s[cy * rw + cx]; };
        auto gx = [&](const float *s, int l, int rr, int cy) { return 0.5f * (at(s, rr, cy) - at(s, l, cy)); };
        auto gy = [&](const float *s, int cx, int u, int d) { return 0.5f * (at(s, cx, d) - at(s, cx, u)); };
        const float z2 = r.zeta * r.zeta, e2 = r.eps * r.eps;
        float sc_t = 0.f, sg_t = 0.f;           // arguments of the two penalisers
        float c11 = 0.f, c12 = 0.f, c22 = 0.f, cb1 = 0.f, cb2 = 0.f;   // colour parts
        float g11 = 0.f, g12 = 0.f, g22 = 0.f, gb1 = 0.f, gb2 = 0.f;   // gradient parts
        float grad1 = 0.f;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const float *i1 = s + c * n, *i2 = s + (C + c) * n;
            const float g1x = gx(i1, jl, jr, jy), g1y = gy(i1, jx, ju, jd);
            const float g2x = gx(i2, jl, jr, jy), g2y = gy(i2, jx, ju, jd);
            grad1 += g1x * g1x + g1y * g1y;
            // colour constancy
            const float Ix = 0.5f * (g1x + g2x), Iy = 0.5f * (g1y + g2y);
            const float Iz = at(i2, jx, jy) - at(i1, jx, jy);
            const float t0 = 1.f / (Ix * Ix + Iy * Iy + z2);
            sc_t += t0 * Iz * Iz;
            c11 += t0 * Ix * Ix; c12 += t0 * Ix * Iy; c22 += t0 * Iy * Iy;
            cb1 += t0 * Ix * Iz; cb2 += t0 * Iy * Iz;
            // gradient constancy: derivatives of the gradient images
            const float Ixx = 0.5f * (0.5f * (gx(i1, xrl, xrr, jy) - gx(i1, xll, xlr, jy)) +
                                      0.5f * (gx(i2, xrl, xrr, jy) - gx(i2, xll, xlr, jy)));
            const float Ixy = 0.5f * (0.5f * (gx(i1, jl, jr, jd) - gx(i1, jl, jr, ju)) +
                                      0.5f * (gx(i2, jl, jr, jd) - gx(i2, jl, jr, ju)));
            const float Iyx = 0.5f * (0.5f * (gy(i1, jr, ju, jd) - gy(i1, jl, ju, jd)) +
                                      0.5f * (gy(i2, jr, ju, jd) - gy(i2, jl, ju, jd)));
            const float Iyy = 0.5f * (0.5f * (gy(i1, jx, ydu, ydd) - gy(i1, jx, yuu, yud)) +
                                      0.5f * (gy(i2, jx, ydu, ydd) - gy(i2, jx, yuu, yud)));
            const float Ixz = g2x - g1x, Iyz = g2y - g1y;
            const float tx = 1.f / (Ixx * Ixx + Ixy * Ixy + z2);
            const float ty = 1.f / (Iyx * Iyx + Iyy * Iyy + z2);
            sg_t += tx * Ixz * Ixz + ty * Iyz * Iyz;
            g11 += tx * Ixx * Ixx + ty * Iyx * Iyx;
            g12 += tx * Ixx * Ixy + ty * Iyx * Iyy;
            g22 += tx * Ixy * Ixy + ty * Iyy * Iyy;
            gb1 += tx * Ixx * Ixz + ty * Iyx * Iyz;
            gb2 += tx * Ixy * Ixz + ty * Iyy * Iyz;
        }
        const float pc = 0.5f / sqrtf(sc_t + e2);
        const float pg = r.gamma * (0.5f / sqrtf(sg_t + e2));
        // smoothness: alpha(x) Psi'(|grad u|^2 + |grad v|^2), central differences
        const float2 fl = __ldcg(flow + (size_t)y * W + xl), fr = __ldcg(flow + (size_t)y * W + xr);
        const float2 fu = __ldcg(flow + (size_t)yu * W + x), fd = __ldcg(flow + (size_t)yd * W + x);
        const float ux = 0.5f * (fr.x - fl.x), uy = 0.5f * (fd.x - fu.x);
        const float vx = 0.5f * (fr.y - fl.y), vy = 0.5f * (fd.y - fu.y);
        const float alpha = r.alpha0 * expf(-r.kappa * sqrtf(grad1));
        const float phi = alpha * (0.5f / sqrtf(ux * ux + uy * uy + vx * vx + vy * vy + e2));
        o.a[p] = make_float4(pc * c11 + pg * g11, pc * c12 + pg * g12, pc * c22 + pg * g22, pc * cb1 + pg * gb1);
        o.b[p] = make_float2(pc * cb2 + pg * gb2, phi);
    }
}

// The same for a whole frame.
constexpr int CT_W = 32, CT_H = 8;
template <int C>
__global__ void __launch_bounds__(CT_W * CT_H) coeff_kernel(const float *__restrict__ I1, const float *__restrict__ I2,
                                                            const float2 *flow, int W, int H, RefineArgs r,
                                                            RefineScratch o) {
    __shared__ float s[2 * C * (CT_W + 4) * (CT_H + 4)];
    const int across = (W + CT_W - 1) / CT_W;
    coeff_tile<C>(I1, I2, flow, W, H, r, o, (int)(blockIdx.x % across) * CT_W, (int)(blockIdx.x / across) * CT_H,
                  CT_W, CT_H, s);
}

// ---------------------------------------------------------------------------
// Red-black SOR, point-coupled: the 2x2 system of (du, dv) at a pixel is
// solved exactly from the current neighbours and over-relaxed.
// ---------------------------------------------------------------------------
// A CTA holds a core of cw x ch pixels and SOR_H pixels around it on chip.
// Cells on the region's outer ring are never updated; a wrong value spreads
// inward by one pixel per half-sweep, so after SOR_H half-sweeps the core
// holds exactly what the half-sweeps over the whole image would give (each
// update is the same arithmetic on the same values).  Then the CTAs exchange
// the updates of the cells near their cores' edges.
//
// Cells of a colour are consecutive, row by row: cell (r, c) is entry
// r * half + c / 2 of its colour's arrays, and thread t owns the entries t,
// t + threads, t + 2 threads of either colour.  What only the owner needs and
// what an update changes stays in its registers; neighbours are read from
// shared memory (18 wavefronts of 32 words per 32 updates).
//
// 1024 x 436, three channels, 5 iterations of 60 half-sweeps: 654 us; before,
// a launch per six half-sweeps that loaded 1.9 times its core from global
// memory, two divisions per update and a launch each for warp, coefficients
// and update: 1930 us and 190 us between launches.  An iteration now: 24 us
// coefficients, 10 us to load the tiles, 1.0 us per half-sweep (what bounds it:
// instruction issue, ~100 per update), 4.4 us per exchange (latency through
// L2).  Also measured: four half-sweeps per exchange, two CTAs an SM, 683 us;
// strips of six cells of a column per thread (vertical neighbours in
// registers) spill: 1.2 - 2.5 us per half-sweep; flags and fences instead of
// tagged words 6 us per exchange; a launch each for the parts 760 us.
constexpr int PER_COLOUR = 3;   // cells of a colour per thread
constexpr int SOR_THREADS = 768;
constexpr int SOR_PER_SM = 1;   // CTAs an SM
constexpr int SOR_CELLS = PER_COLOUR * SOR_THREADS;   // of a colour
constexpr int BATCH = 3;        // cells around the core that a thread fetches at once
constexpr unsigned long long SOR_WAIT_NS = 1000000000ull;   // 1 s
constexpr int SEND = 1 << 30, RECEIVE = 1 << 29, ENTRY = RECEIVE - 1;
struct SorShared {
    float4 own[2][SOR_CELLS];    // u, v, b1, b2
    float2 sum[2][SOR_CELLS];    // u + du, v + dv
    float2 d[2][SOR_CELLS];      // du, dv of cells that other CTAs own, as they arrive
    float right[2][SOR_CELLS];   // weight of the edge to the right (first: phi)
    float down[2][SOR_CELLS];    // and downwards
};

struct SorGrid {
    int cw, ch, tiles_x, tiles_y;   // cores
    int half, rh;                   // region: 2 half x rh cells
};

struct SorCell {
    float a, b, d, inv;   // system a b; b d, and 1 / det (0: not updated, < 0: divide)
    float du, dv;
};

// Whether a wait is to end: `limit` ns after its first call (*t0 = 0), or when
// another CTA has given up.
__device__ __noinline__ bool sor_gives_up(unsigned long long *t0, unsigned *error, RunState *st,
                                          unsigned long long limit) {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    if (*t0 == 0) *t0 = t;
    if (t - *t0 <= limit && *(volatile unsigned *)error == 0u) return false;
    atomicExch(error, 1u);
    set_status(st, EPIC_ERR_TIMEOUT);
    return true;
}

// Waits until the neighbouring tiles' progress is `want` at least (false in
// every thread: gave up).
__device__ bool sor_wait(const SorGrid &g, unsigned *progress, unsigned want, RunState *st,
                         unsigned long long limit = SOR_WAIT_NS) {
    const int k = threadIdx.x;
    bool failed = false;
    if (k < 8) {
        const int x = (int)blockIdx.x % g.tiles_x + (k < 3 ? k - 1 : k < 5 ? 2 * k - 7 : k - 6);
        const int y = (int)blockIdx.x / g.tiles_x + (k < 3 ? -1 : k < 5 ? 0 : 1);
        if (x >= 0 && x < g.tiles_x && y >= 0 && y < g.tiles_y) {
            unsigned long long t0 = 0;
            for (int n = 1; ld_acquire(progress + y * g.tiles_x + x) < want; ++n)
                if ((n & 63) == 0 && sor_gives_up(&t0, progress + g.tiles_x * g.tiles_y, st, limit)) {
                    failed = true;
                    break;
                }
        }
    }
    return __syncthreads_or(failed) == 0;
}

// A cell's update with the round that wrote it beside either half, so that the
// reader needs no flag and the writer no fence.
__device__ __forceinline__ void put_tagged(ulonglong2 *p, float du, float dv, unsigned tag) {
    const unsigned long long t = (unsigned long long)tag << 32;
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(t | __float_as_uint(du)),
                 "l"(t | __float_as_uint(dv))
                 : "memory");
}
__device__ __forceinline__ void get_tagged(const ulonglong2 *p, ulonglong2 *v) {
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(v->x), "=l"(v->y) : "l"(p) : "memory");
}
// Reads *p into *v until it carries the tag (false: gave up).
__device__ __forceinline__ bool await_tagged(const ulonglong2 *p, unsigned tag, ulonglong2 *v, unsigned *error,
                                             RunState *st, unsigned long long limit = SOR_WAIT_NS) {
    unsigned long long t0 = 0;
    for (int m = 1; (unsigned)(v->x >> 32) != tag || (unsigned)(v->y >> 32) != tag; ++m) {
        if ((m & 63) == 0 && sor_gives_up(&t0, error, st, limit)) return false;
        get_tagged(p, v);
    }
    return true;
}

// This CTA's writes, by every thread, are done up to step `step`.
__device__ void sor_post(unsigned *progress, unsigned step) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();   // (cumulative: the CTA's writes, ordered by the barrier)
        atomicExch(progress + blockIdx.x, step);
    }
}

// C > 0: a whole refinement of frames with C channels in one cooperative
// launch, a CTA per tile.  C = 0: SOR_H half-sweeps at most of one linear
// system, from updates din (null: zero) to dout.
template <int C>
__global__ void __launch_bounds__(SOR_THREADS, SOR_PER_SM)
    sor_kernel(const float *__restrict__ I1, const float *__restrict__ I2, float2 *flow, RefineArgs ra,
               RefineScratch x, SorGrid g, int W, int H, int nhalf, const float2 *din, float2 *dout, RunState *st) {
    constexpr bool ROUNDS = C > 0;
    const float omega = ra.omega;
    extern __shared__ __align__(16) unsigned char smem[];
    SorShared &sh = *reinterpret_cast<SorShared *>(smem);
    const int tid = threadIdx.x, NT = blockDim.x, half = g.half, n = half * g.rh;
    const int rx0 = (int)blockIdx.x % g.tiles_x * g.cw - SOR_H, ry0 = (int)blockIdx.x / g.tiles_x * g.ch - SOR_H;
    const int par = (rx0 + ry0) & 1;
    const int r1 = SOR_H + g.ch, c1 = SOR_H + g.cw;   // of the core
    SorCell cell[2][PER_COLOUR];
    int code[2][PER_COLOUR];   // 2 * entry + odd column, SEND, RECEIVE
    const int iterations = ROUNDS ? ra.iterations : 1;
    unsigned tag = 0;
    for (int it = 0; it < iterations; ++it) {
        if constexpr (ROUNDS) {
            // (the flow around the core is the neighbours')
            if (it > 0 && !sor_wait(g, x.progress, 3u * it, st)) return;
            coeff_tile<C>(I1, I2, flow, W, H, ra, x, rx0 + SOR_H, ry0 + SOR_H, g.cw, g.ch, reinterpret_cast<float *>(smem));
            sor_post(x.progress, 3u * it + 1u);
            if (!sor_wait(g, x.progress, 3u * it + 1u, st)) return;
        }
        const unsigned inv_half = 0xFFFFFFFFu / (unsigned)half + 1;   // (entry * inv_half) >> 32 is its row
        // f(colour, slot, entry, row, column, X, Y) for the thread's cells in the image
        auto cells = [&](auto &&f) {
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int j = 0; j < PER_COLOUR; ++j) {
                    const int k = tid + j * NT;
                    if (k >= n) continue;
                    const int r = __umulhi(k, inv_half), c = 2 * (k - r * half) + ((q + par + r) & 1);
                    const int X = rx0 + c, Y = ry0 + r;
                    if (X >= 0 && X < W && Y >= 0 && Y < H) f(q, j, k, r, c, X, Y);
                }
        };
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int j = 0; j < PER_COLOUR; ++j) {
                cell[q][j] = SorCell{0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
                code[q][j] = 0;
                const int k = tid + j * NT;
                if (k >= n) continue;
                sh.sum[q][k] = make_float2(0.f, 0.f);
                sh.right[q][k] = sh.down[q][k] = 0.f;
            }
        cells([&](int q, int j, int k, int r, int c, int X, int Y) {
            SorCell &z = cell[q][j];
            const size_t p = (size_t)Y * W + X;
            const float4 A = __ldcg(x.a + p);
            const float2 B = __ldcg(x.b + p), f = __ldcg(flow + p);
            if (!ROUNDS && din) {
                const float2 d = din[p];
                z.du = d.x;
                z.dv = d.y;
            }
            z.a = A.x;
            z.b = A.y;
            z.d = A.z;
            sh.own[q][k] = make_float4(f.x, f.y, A.w, B.x);
            sh.sum[q][k] = make_float2(f.x + z.du, f.y + z.dv);
            sh.right[q][k] = B.y;
        });
        __syncthreads();
        float wr[2][PER_COLOUR], wd[2][PER_COLOUR];
        cells([&](int q, int j, int k, int r, int c, int X, int Y) {
            wr[q][j] = wd[q][j] = 0.f;
            SorCell &z = cell[q][j];
            const float phi = sh.right[q][k];
            const int odd = c & 1, kl = k - 1 + odd;
            float S = 0.f;   // right, left, down, up
            if (X + 1 < W && c < 2 * half - 1) S += wr[q][j] = 0.5f * (phi + sh.right[1 - q][kl + 1]);
            if (X > 0 && c > 0) S += 0.5f * (phi + sh.right[1 - q][kl]);
            if (Y + 1 < H && r < g.rh - 1) S += wd[q][j] = 0.5f * (phi + sh.right[1 - q][k + half]);
            if (Y > 0 && r > 0) S += 0.5f * (phi + sh.right[1 - q][k - half]);
            z.a += S;
            z.d += S;
            const float det = z.a * z.d - z.b * z.b;
            const bool core = r >= SOR_H && r < r1 && c >= SOR_H && c < c1;
            code[q][j] = 2 * k + odd;
            if (!core) code[q][j] |= RECEIVE;
            else if (r < 2 * SOR_H || r >= g.ch || c < 2 * SOR_H || c >= g.cw) code[q][j] |= SEND;
            // (an inverse whose residuals are normal numbers; otherwise divide)
            if (r > 0 && c > 0 && r < g.rh - 1 && c < 2 * half - 1)
                z.inv = !(det > 0.f) ? 0.f : det > 1e-18f && det < 1e18f ? 1.f / det : -1.f;
        });
        __syncthreads();
        cells([&](int q, int j, int k, int r, int c, int X, int Y) {
            sh.right[q][k] = wr[q][j];
            sh.down[q][k] = wd[q][j];
        });
        if (ROUNDS) sor_post(x.progress, 3u * it + 2u);   // (the flow of this region is read)
        else __syncthreads();
        const float keep = 1.f - omega;
        auto half_sweep = [&](auto colour) {
            constexpr int q = decltype(colour)::value;
#pragma unroll
            for (int j = 0; j < PER_COLOUR; ++j) {
                SorCell &z = cell[q][j];
                if (z.inv == 0.f) continue;
                // (addresses are computed anew: kept across half-sweeps, they would spill)
                asm volatile("" : "+r"(code[q][j]));
                const int k = (code[q][j] & ENTRY) >> 1, kl = ((code[q][j] + 1) & ENTRY) / 2 - 1;
                const float4 o = sh.own[q][k];
                float r1 = 0.f, r2 = 0.f;
                auto nb = [&](float2 t, float w) {   // right, left, down, up
                    r1 += w * (t.x - o.x);
                    r2 += w * (t.y - o.y);
                };
                nb(sh.sum[1 - q][kl + 1], sh.right[q][k]);
                nb(sh.sum[1 - q][kl], sh.right[1 - q][kl]);
                nb(sh.sum[1 - q][k + half], sh.down[q][k]);
                nb(sh.sum[1 - q][k - half], sh.down[1 - q][k - half]);
                r1 -= o.z;
                r2 -= o.w;
                const float nu = z.d * r1 - z.b * r2, nv = z.a * r2 - z.b * r1;
                const float det = z.a * z.d - z.b * z.b;
                float qu, qv;
                if (z.inv > 0.f) {
                    qu = quotient(nu, det, z.inv);
                    qv = quotient(nv, det, z.inv);
                } else {
                    qu = nu / det;
                    qv = nv / det;
                }
                z.du = keep * z.du + omega * qu;
                z.dv = keep * z.dv + omega * qv;
                sh.sum[q][k] = make_float2(o.x + z.du, o.y + z.dv);
            }
            __syncthreads();
        };
        // the cells around the core that this thread fetches: 2 * entry + colour
        // (-1: none) and pixel
        int to[BATCH];
        unsigned from[BATCH];
        if (ROUNDS) {
            const int band = 2 * SOR_H * 2 * half, around = band + 2 * SOR_H * g.ch;
#pragma unroll
            for (int k = 0; k < BATCH; ++k) {
                const int h = tid + k * NT;
                int hr, hc;
                if (h < band) {
                    hr = h / (2 * half);
                    hc = h - hr * 2 * half;
                    if (hr >= SOR_H) hr += g.ch;
                } else {
                    hr = (h - band) / (2 * SOR_H);
                    hc = h - band - hr * 2 * SOR_H;
                    if (hc >= SOR_H) hc += g.cw;
                    hr += SOR_H;
                }
                const int hx = rx0 + hc, hy = ry0 + hr;
                const bool in = h < around && hx >= 0 && hx < W && hy >= 0 && hy < H;
                to[k] = in ? 2 * (hr * half + (hc >> 1)) + ((hr + hc + par) & 1) : -1;
                from[k] = in ? (unsigned)(hy * W + hx) : 0u;
            }
        }
        for (int done = 0;;) {
            const int nh = min(SOR_H, nhalf - done);
            for (int h = 0; h < nh; h += 2) {   // (nhalf is even)
                half_sweep(std::integral_constant<int, 0>{});
                half_sweep(std::integral_constant<int, 1>{});
            }
            done += nh;
            if (!ROUNDS || done >= nhalf) break;
            // exchange: the core's cells near its edges out, the cells around it in.
            // Two buffers in turn: a neighbour writes a third round only when it
            // has read the second, which this CTA writes when it has read the first.
            ulonglong2 *buf = x.swap[tag & 1];
            ++tag;
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int j = 0; j < PER_COLOUR; ++j) {
                    if (!(code[q][j] & SEND)) continue;
                    const int k = tid + j * NT, r = __umulhi(k, inv_half), c = 2 * (k - r * half) + (code[q][j] & 1);
                    put_tagged(buf + (ry0 + r) * W + rx0 + c, cell[q][j].du, cell[q][j].dv, tag);
                }
            bool failed = false;
            ulonglong2 v[BATCH];
#pragma unroll
            for (int k = 0; k < BATCH; ++k)   // (all loads before any is looked at)
                if (to[k] >= 0) get_tagged(buf + from[k], &v[k]);
#pragma unroll
            for (int k = 0; k < BATCH; ++k) {
                if (to[k] < 0) continue;
                if (!await_tagged(buf + from[k], tag, &v[k], x.progress + g.tiles_x * g.tiles_y, st)) failed = true;
                const float2 d = make_float2(__uint_as_float((unsigned)v[k].x), __uint_as_float((unsigned)v[k].y));
                const int q = to[k] & 1, e = to[k] >> 1;
                const float4 o = sh.own[q][e];
                sh.d[q][e] = d;
                sh.sum[q][e] = make_float2(o.x + d.x, o.y + d.y);
            }
            if (__syncthreads_or(failed)) return;
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int j = 0; j < PER_COLOUR; ++j) {
                    if (!(code[q][j] & RECEIVE)) continue;
                    const float2 d = sh.d[q][tid + j * NT];
                    cell[q][j].du = d.x;
                    cell[q][j].dv = d.y;
                }
        }
        // the core
        if (ROUNDS && !sor_wait(g, x.progress, 3u * it + 2u, st)) return;   // (its flow is read by all that need it)
        cells([&](int q, int j, int k, int r, int c, int X, int Y) {
            if (r < SOR_H || r >= r1 || c < SOR_H || c >= c1) return;
            const size_t p = (size_t)Y * W + X;
            if (ROUNDS) flow[p] = sh.sum[q][k];
            else dout[p] = make_float2(cell[q][j].du, cell[q][j].dv);
        });
        if (ROUNDS && it + 1 < iterations) sor_post(x.progress, 3u * it + 3u);
    }
}

// Self-test of this kernel's waits (see epic_selftest_wait_timeout): nobody makes
// progress and nobody sends an update.
__device__ unsigned selftest_progress[3];
__device__ ulonglong2 selftest_update;
__global__ void refine_wait_selftest_kernel(RunState *st, int which, unsigned long long limit_ns) {
    if (threadIdx.x < 3) selftest_progress[threadIdx.x] = 0;
    __threadfence();
    __syncthreads();
    if (which == 5) {
        sor_wait(SorGrid{8, 8, 2, 1, 10, 20}, selftest_progress, 1u, st, limit_ns);
    } else if (threadIdx.x == 0) {
        ulonglong2 v;
        get_tagged(&selftest_update, &v);
        await_tagged(&selftest_update, 1u, &v, selftest_progress + 2, st, limit_ns);
    }
}

__global__ void update_kernel(float *__restrict__ flow, const float *__restrict__ d, long long n2) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n2;
         i += (long long)gridDim.x * blockDim.x)
        flow[i] += d[i];
}

int even(int v) { return (v + 1) & ~1; }

// A thread per PER_COLOUR cells of a colour and BATCH cells around the core.
int sor_threads(const SorGrid &g) {
    const int cells = g.half * g.rh, around = 2 * cells - g.cw * g.ch;
    return (std::max((cells + PER_COLOUR - 1) / PER_COLOUR, (around + BATCH - 1) / BATCH) + 31) / 32 * 32;
}

SorGrid sor_grid_of(int cw, int ch, int W, int H) {
    return SorGrid{cw, ch, (W + cw - 1) / cw, (H + ch - 1) / ch, cw / 2 + SOR_H, ch + 2 * SOR_H};
}

// Cores that cover the frame in one wave of CTAs with the fewest threads;
// false if that takes more than SOR_THREADS.  A
// core is at least SOR_H wide and high (the cells around it are its eight
// neighbours').
//
// (1024 x 436 takes 668 us in one wave, 970 us with a launch per six
// half-sweeps; 128 x 256 takes 340 and 784 us.)
bool sor_one_wave(int W, int H, int num_sms, SorGrid *best) {
    int fewest = SOR_THREADS + 1;
    const int most = std::min(SOR_PER_SM * num_sms, SOR_MAX_TILES);
    for (int tx = 1; tx <= most; ++tx) {
        const int cw = std::max(even((W + tx - 1) / tx), SOR_H);
        const int ty = most / ((W + cw - 1) / cw);
        if (ty < 1) continue;
        const SorGrid g = sor_grid_of(cw, std::max((H + ty - 1) / ty, SOR_H), W, H);
        if ((long long)g.half * g.rh <= SOR_CELLS && sor_threads(g) < fewest) {
            fewest = sor_threads(g);
            *best = g;
        }
    }
    return fewest <= SOR_THREADS;
}

size_t rf_align(size_t b) { return (b + 255) / 256 * 256; }

template <int C>
void launch_coeff(const float *I1, const float *I2, int H, int W, const float *flow, const RefineArgs &r,
                  const RefineScratch &x, cudaStream_t stream) {
    const long long tiles = (long long)((W + CT_W - 1) / CT_W) * ((H + CT_H - 1) / CT_H);
    coeff_kernel<C><<<(unsigned)tiles, CT_W * CT_H, 0, stream>>>(I1, I2, reinterpret_cast<const float2 *>(flow), W,
                                                                 H, r, x);
}

}  // namespace

cudaError_t launch_refine_wait_selftest(RunState *st, int which, unsigned long long limit_ns, cudaStream_t stream) {
    refine_wait_selftest_kernel<<<1, 32, 0, stream>>>(st, which, limit_ns);
    return cudaGetLastError();
}

size_t refine_scratch_bytes(int H, int W) {
    const size_t P = (size_t)H * W;
    return rf_align(P * sizeof(float4)) + rf_align(P * sizeof(float2)) + 2 * rf_align(P * sizeof(ulonglong2)) +
           rf_align((SOR_MAX_TILES + 1) * sizeof(unsigned));
}

static cudaError_t refine_frames(const float *I1, const float *I2, int H, int W, int C, float *flow,
                          const RefineArgs &r, void *scratch, int num_sms, RunState *state, cudaStream_t stream, bool one_launch) {
    const size_t P = (size_t)H * W;
    char *base = static_cast<char *>(scratch);
    auto take = [&](size_t bytes) {
        char *p = base;
        base += rf_align(bytes);
        return p;
    };
    RefineScratch x;
    x.a = reinterpret_cast<float4 *>(take(P * sizeof(float4)));
    x.b = reinterpret_cast<float2 *>(take(P * sizeof(float2)));
    x.swap[0] = reinterpret_cast<ulonglong2 *>(take(P * sizeof(ulonglong2)));
    x.swap[1] = reinterpret_cast<ulonglong2 *>(take(P * sizeof(ulonglong2)));
    x.progress = reinterpret_cast<unsigned *>(take((SOR_MAX_TILES + 1) * sizeof(unsigned)));
    SorGrid g;
    const bool one_wave = one_launch && sor_one_wave(W, H, num_sms, &g);
    if (!one_wave) g = sor_grid_of(64, 48, W, H);
    const int threads = sor_threads(g);
    const int nhalf = 2 * r.sor_iterations;
    float2 *const f2 = reinterpret_cast<float2 *>(flow);
    cudaError_t e;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(g.tiles_x * g.tiles_y));
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = sizeof(SorShared);
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = one_wave ? 1 : 0;
    auto *sor = !one_wave ? sor_kernel<0> : C == 1 ? sor_kernel<1> : C == 2 ? sor_kernel<2> : C == 3 ? sor_kernel<3>
                                                                                           : sor_kernel<4>;
    if ((e = cudaFuncSetAttribute(sor, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SorShared))) !=
        cudaSuccess)
        return e;
    auto launch = [&](int half_sweeps, const float2 *din, float2 *dout) {
        return cudaLaunchKernelEx(&cfg, sor, I1, I2, f2, r, x, g, W, H, half_sweeps, din, dout, state);
    };
    if (one_wave) {
        if (r.iterations == 0) return cudaSuccess;
        // (no tag and no progress of an earlier refinement)
        if ((e = cudaMemsetAsync(x.swap[0], 0, base - reinterpret_cast<char *>(x.swap[0]), stream)) != cudaSuccess)
            return e;
        return launch(nhalf, nullptr, nullptr);
    }
    for (int it = 0; it < r.iterations; ++it) {
        switch (C) {
            case 1: launch_coeff<1>(I1, I2, H, W, flow, r, x, stream); break;
            case 2: launch_coeff<2>(I1, I2, H, W, flow, r, x, stream); break;
            case 3: launch_coeff<3>(I1, I2, H, W, flow, r, x, stream); break;
            default: launch_coeff<4>(I1, I2, H, W, flow, r, x, stream);
        }
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        int cur = 1;   // the buffer of the latest update
        for (int done = 0; done < nhalf; done += SOR_H, cur ^= 1)
            if ((e = launch(std::min(SOR_H, nhalf - done), done ? x.d[cur] : nullptr, x.d[cur ^ 1])) != cudaSuccess)
                return e;
        if (nhalf > 0) {
            const long long blocks = std::min<long long>((2 * (long long)P + 255) / 256, 8LL * num_sms);
            update_kernel<<<(unsigned)blocks, 256, 0, stream>>>(flow, reinterpret_cast<const float *>(x.d[cur]),
                                                                2 * (long long)P);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
    }
    return cudaSuccess;
}

cudaError_t launch_refine(const float *I1, const float *I2, int H, int W, int C, float *flow,
                          const RefineArgs &r, void *scratch, int num_sms, RunState *state, cudaStream_t stream) {
    cudaError_t e = refine_frames(I1, I2, H, W, C, flow, r, scratch, num_sms, state, stream, true);
    if (e != cudaErrorCooperativeLaunchTooLarge) return e;
    // a context with a part of the GPU's SMs
    cudaGetLastError();
    return refine_frames(I1, I2, H, W, C, flow, r, scratch, num_sms, state, stream, false);
}

}  // namespace epic
