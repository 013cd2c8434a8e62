// Cost map from the image gradient (Table 2, the "||grad_2 I||_2" contour
// row): C(p) = floor + sqrt(sum_c gx_c^2 + gy_c^2) with central differences
// gx = (I(x+1) - I(x-1)) / 2 on the edge-replicated image.
//
// A stack of frames [F][H][W][channels] float32 is processed in one launch;
// each frame's borders are its own.  The algorithmic traffic is one read of
// the image and one write of the cost (channels * 4 + 4 bytes per pixel), and
// HBM bounds it.
//
// A warp walks down a strip of columns; a lane holds a few neighbouring
// pixels of the rows above, at and below it in registers, with the loads of
// the next rows in flight, so every input byte is loaded about once
// (the two lanes at the strip's ends load the columns next to it for the
// others, the rows at its ends come twice, both from L2), with 16-byte loads
// where base and pitch allow them, and nothing passes through shared memory.
// 32 frames of 1024 x 436 x 3: 68 -> 48 us a call, 3.35 -> 4.73 TB/s of the 6.78
// TB/s that a copy reaches (staging 8-row tiles in shared
// memory between two barriers kept the loads of a CTA from overlapping its
// arithmetic).
#include "epic_internal.cuh"

#include <algorithm>

namespace epic {

namespace {

constexpr int GC_WARPS = 4;        // warps per CTA
// Per channel count: neighbouring pixels a lane holds, the columns of a strip
// (the end lanes' are its neighbours'), and the rows whose loads are in
// flight.  Four channels take two pixels a lane: with four, a lane's rows need
// 122 registers and the kernel is slower (41 against 31 us for 16 frames of
// 1024 x 436 x 4).
template <int CH>
struct Gc {
    static constexpr int PX = CH == 4 ? 2 : 4, COLS = 30 * PX, AHEAD = CH == 1 ? 4 : 2;
};

// A lane's pixels of a row from x0 on (the frame's end columns repeated
// beyond it).  V floats per load: 4 or 2 when every row starts on that
// boundary, else 1.
template <int CH, int V>
__device__ __forceinline__ void gc_load(const float *__restrict__ row, int x0, int W,
                                        float (&o)[Gc<CH>::PX * CH]) {
    if (x0 >= 0 && x0 + Gc<CH>::PX <= W) {
        const float *p = row + (size_t)x0 * CH;
#pragma unroll
        for (int i = 0; i < Gc<CH>::PX * CH; i += V) {
            if constexpr (V == 4) {
                const float4 f = __ldg(reinterpret_cast<const float4 *>(p + i));
                o[i] = f.x;
                o[i + 1] = f.y;
                o[i + 2] = f.z;
                o[i + 3] = f.w;
            } else if constexpr (V == 2) {
                const float2 f = __ldg(reinterpret_cast<const float2 *>(p + i));
                o[i] = f.x;
                o[i + 1] = f.y;
            } else {
                o[i] = __ldg(p + i);
            }
        }
    } else {
#pragma unroll
        for (int i = 0; i < Gc<CH>::PX; ++i)
#pragma unroll
            for (int c = 0; c < CH; ++c)
                o[i * CH + c] = __ldg(row + (size_t)min(max(x0 + i, 0), W - 1) * CH + c);
    }
}

template <int CH, int V>
__global__ void __launch_bounds__(GC_WARPS * 32) gradcost_kernel(const float *__restrict__ img, int H,
                                                                 int W, int strips_x, int rows,
                                                                 int chunks, long long strips,
                                                                 float floor_, bool vec_out,
                                                                 float *__restrict__ C) {
    const int lane = threadIdx.x & 31;
    // (whole warps leave: the shuffles below are full)
    const long long s = blockIdx.x * (long long)GC_WARPS + (threadIdx.x >> 5);
    if (s >= strips) return;
    const int sx = (int)(s % strips_x);
    const long long t = s / strips_x;
    const int y0 = (int)(t % chunks) * rows, y1 = min(H, y0 + rows);
    const size_t f = (size_t)(t / chunks);
    const int x0 = sx * Gc<CH>::COLS + (lane - 1) * Gc<CH>::PX;
    const bool mine = lane > 0 && lane < 31;
    const float *fr = img + f * H * W * CH;
    float *out = C + f * H * W;
    const size_t pitch = (size_t)W * CH;
    auto row = [&](int y) { return fr + pitch * (size_t)min(max(y, 0), H - 1); };
    // rows y - 1, y, y + 1 and those in flight in r[]
    constexpr int NR = 3 + Gc<CH>::AHEAD;
    float r[NR][Gc<CH>::PX * CH];
#pragma unroll
    for (int i = 0; i < NR - 1; ++i) gc_load<CH, V>(row(y0 - 1 + i), x0, W, r[i]);
    for (int yb = y0; yb < y1; yb += NR) {
        // (the rows turn through r[] once per NR steps: no copies)
#pragma unroll
        for (int k = 0; k < NR; ++k) {
            const int y = yb + k;
            if (y >= y1) break;
            if (y + 1 + Gc<CH>::AHEAD <= y1) gc_load<CH, V>(row(y + 1 + Gc<CH>::AHEAD), x0, W, r[(k + NR - 1) % NR]);
            const float(&up)[Gc<CH>::PX * CH] = r[k], (&mid)[Gc<CH>::PX * CH] = r[(k + 1) % NR],
                       (&dn)[Gc<CH>::PX * CH] = r[(k + 2) % NR];
            float s2[Gc<CH>::PX] = {};
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                const float left = __shfl_up_sync(0xffffffffu, mid[(Gc<CH>::PX - 1) * CH + c], 1);
                const float right = __shfl_down_sync(0xffffffffu, mid[c], 1);
#pragma unroll
                for (int i = 0; i < Gc<CH>::PX; ++i) {
                    const float a = i ? mid[(i - 1) * CH + c] : left;
                    const float b = i < Gc<CH>::PX - 1 ? mid[(i + 1) * CH + c] : right;
                    const float gx = __fmul_rn(__fsub_rn(b, a), 0.5f);
                    const float gy = __fmul_rn(__fsub_rn(dn[i * CH + c], up[i * CH + c]), 0.5f);
                    s2[i] = __fmaf_rn(gx, gx, s2[i]);
                    s2[i] = __fmaf_rn(gy, gy, s2[i]);
                }
            }
            float o[Gc<CH>::PX];
#pragma unroll
            for (int i = 0; i < Gc<CH>::PX; ++i) o[i] = __fadd_rn(floor_, __fsqrt_rn(s2[i]));
            float *dst = out + (size_t)y * W + x0;
            if (!mine) {
            } else if (x0 + Gc<CH>::PX <= W && vec_out) {
                if constexpr (Gc<CH>::PX == 4)
                    __stcs(reinterpret_cast<float4 *>(dst), make_float4(o[0], o[1], o[2], o[3]));
                else
                    __stcs(reinterpret_cast<float2 *>(dst), make_float2(o[0], o[1]));
            } else {
#pragma unroll
                for (int i = 0; i < Gc<CH>::PX; ++i)
                    if (x0 + i < W) __stcs(dst + i, o[i]);
            }
        }
    }
}

template <int CH, int V>
cudaError_t gradcost_launch(const float *img, int F, int H, int W, float floor_, float *C,
                            int num_sms, cudaStream_t stream) {
    // (a property of the kernel, asked for once: the query takes longer than a
    // launch)
    static const int per_sm = [] {
        int n = 0;
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, gradcost_kernel<CH, V>,
                                                             GC_WARPS * 32, 0) == cudaSuccess
                   ? std::max(n, 1)
                   : 1;
    }();
    const long long resident = (long long)num_sms * per_sm * GC_WARPS;
    const int strips_x = (W + Gc<CH>::COLS - 1) / Gc<CH>::COLS;
    // strip height: the number of waves of resident warps, one to eight, that
    // takes the fewest rows in all (a strip loads two rows of its neighbours'
    // and starts with nothing in flight: about four rows' time)
    int rows = H, chunks = 1;
    long long best = 0;
    for (int waves = 1; waves <= 8; ++waves) {
        const long long c = std::min<long long>(std::max(1LL, waves * resident / ((long long)F * strips_x)), H);
        const int r = (int)((H + c - 1) / c), n = (H + r - 1) / r;
        const long long cost = ((long long)F * strips_x * n + resident - 1) / resident * (r + 4);
        if (waves == 1 || cost < best) {
            best = cost;
            rows = r;
            chunks = n;
        }
    }
    const long long strips = (long long)F * chunks * strips_x;
    const long long blocks = (strips + GC_WARPS - 1) / GC_WARPS;
    if (blocks > 2147483647LL) return cudaErrorInvalidValue;
    const bool vec_out = W % 4 == 0 && ((uintptr_t)C & 15) == 0;
    gradcost_kernel<CH, V><<<(unsigned)blocks, GC_WARPS * 32, 0, stream>>>(
        img, H, W, strips_x, rows, chunks, strips, floor_, vec_out, C);
    return cudaGetLastError();
}

template <int CH>
cudaError_t gradcost_channels(const float *img, int F, int H, int W, float floor_, float *C,
                              int num_sms, cudaStream_t stream) {
    // every row (and a lane's first pixel in it) on a 16- or 8-byte boundary?
    const size_t pitch = (size_t)W * CH * 4;
    const uintptr_t a = (uintptr_t)img | pitch;
    if (a % 16 == 0) return gradcost_launch<CH, 4>(img, F, H, W, floor_, C, num_sms, stream);
    if (a % 8 == 0) return gradcost_launch<CH, 2>(img, F, H, W, floor_, C, num_sms, stream);
    return gradcost_launch<CH, 1>(img, F, H, W, floor_, C, num_sms, stream);
}

}  // namespace

cudaError_t launch_gradcost(const float *img, int F, int H, int W, int channels, float floor_,
                            float *C, int num_sms, cudaStream_t stream) {
    switch (channels) {
    case 1: return gradcost_channels<1>(img, F, H, W, floor_, C, num_sms, stream);
    case 3: return gradcost_channels<3>(img, F, H, W, floor_, C, num_sms, stream);
    case 4: return gradcost_channels<4>(img, F, H, W, floor_, C, num_sms, stream);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace epic
