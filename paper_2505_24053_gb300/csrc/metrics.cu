// metrics.cu -- evaluation of a native-camera image against a reference image
// (the paper's evaluation of renders reprojected to the native fisheye image):
// per region, the sum of squared errors over pixels and channels, the sum of
// the per-pixel SSIM (mean over the three channels) and the pixel count.
//
// SSIM (Wang et al. 2004, as 3DGS-style evaluations compute it): local means,
// variances and covariance under an 11 x 11 Gaussian window (sigma 1.5,
// normalised), zero padding at the image border, C1 = 0.01^2, C2 = 0.03^2 for
// values in [0, 1]. A block takes a 32 x 16 tile: the tile and a 5-pixel halo of
// both images are staged in shared memory as pairs (x, y), the window is applied per
// channel as a horizontal then a vertical 11-tap pass to the five quantities x, y, x^2,
// y^2, xy, and the block's sums per region are added to FP64 accumulators with one
// atomic each. Bound by issued instructions: a thread takes four neighbouring columns
// (14 loads for 44 taps), then two rows, with packed arithmetic for the pairs, and the
// taps stay in registers. (1280 x 960, two regions: 49 us, where a thread per output
// that loaded every tap took 75.)
#include "geer_internal.cuh"

namespace geer {
namespace {

constexpr int kMW = 32, kMH = 16;                         // output tile
constexpr int kHalo = 5, kTaps = 2 * kHalo + 1;           // window radius, taps
constexpr int kInW = kMW + 2 * kHalo, kInH = kMH + 2 * kHalo;  // staged tile
constexpr int kMThreads = 256;
constexpr int kMaxRegions = 8;
static_assert(kMW == 32 && kMW * kMH == 2 * kMThreads, "a thread per column and two rows in the vertical pass");
static_assert(kInH * kMW / 4 <= kMThreads && kInW % 2 == 0, "a thread per four columns in the horizontal pass");

// The five quantities' window sums: x and y, x^2 and y^2, xy.
struct Moments {
    float2 xy, xx;
    float c;
};

__global__ void __launch_bounds__(kMThreads) k_image_metrics(const float *__restrict__ pred,
                                                             const float *__restrict__ gt, int w, int h,
                                                             const uint8_t *__restrict__ regions, int nreg,
                                                             double *__restrict__ acc) {
    grid_dep_sync();
    __shared__ __align__(16) float2 s[3][kInH][kInW];  // (pred, gt)
    __shared__ __align__(16) float2 h_xy[kInH][kMW], h_xx[kInH][kMW];
    __shared__ __align__(16) float h_c[kInH][kMW];
    __shared__ float red[kMThreads / 32][kMaxRegions][3];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int x0 = (int)blockIdx.x * kMW - kHalo, y0 = (int)blockIdx.y * kMH - kHalo;
    for (int i = tid; i < kInH * kInW; i += kMThreads) {
        const int iy = i / kInW, ix = i - iy * kInW, gx = x0 + ix, gy = y0 + iy;
        const bool in = gx >= 0 && gx < w && gy >= 0 && gy < h;
        const int64_t p = (int64_t)gy * w + gx;
#pragma unroll
        for (int ch = 0; ch < 3; ++ch)
            s[ch][iy][ix] = make_float2(in ? pred[3 * p + ch] : 0.0f, in ? gt[3 * p + ch] : 0.0f);
    }
    // the normalised taps, symmetric: tap k in gw[k <= kHalo ? k : 2 kHalo - k]
    float gw[kHalo + 1];
    {
        const float k = (float)(lane - kHalo), e = expf(-k * k / (2.0f * 1.5f * 1.5f));
        float sum = 0.0f;
#pragma unroll
        for (int t = 0; t < kTaps; ++t) sum += __shfl_sync(0xffffffffu, e, t);
#pragma unroll
        for (int t = 0; t <= kHalo; ++t) gw[t] = __shfl_sync(0xffffffffu, e, t) / sum;
    }
    const auto tap = [&](int k) { return gw[k <= kHalo ? k : 2 * kHalo - k]; };
    const auto add = [&](Moments &m, float g, float2 xy, float2 xx, float c) {
        const float2 gg = make_float2(g, g);
        m.xy = fma2(gg, xy, m.xy);
        m.xx = fma2(gg, xx, m.xx);
        m.c = fmaf(g, c, m.c);
    };
    // the vertical pass's column and first row, their regions and sums
    const int px = lane, py = 2 * warp;
    const int gx = (int)blockIdx.x * kMW + px, gy = (int)blockIdx.y * kMH + py;
    float se[2] = {0.0f, 0.0f}, ss[2] = {0.0f, 0.0f};
    __syncthreads();
#pragma unroll 1
    for (int ch = 0; ch < 3; ++ch) {
        // horizontal pass: rows of the staged tile, four output columns a thread
        if (tid < kInH * (kMW / 4)) {
            const int r = tid / (kMW / 4), c = 4 * (tid - r * (kMW / 4));
            Moments m[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) m[q] = Moments{make_float2(0.0f, 0.0f), make_float2(0.0f, 0.0f), 0.0f};
#pragma unroll
            for (int i = 0; i < kTaps + 3; ++i) {
                const float2 v = s[ch][r][c + i], xx = mul2(v, v);
                const float xy = v.x * v.y;
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (i >= q && i - q < kTaps) add(m[q], tap(i - q), v, xx, xy);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                h_xy[r][c + q] = m[q].xy;
                h_xx[r][c + q] = m[q].xx;
                h_c[r][c + q] = m[q].c;
            }
        }
        __syncthreads();
        // vertical pass and SSIM for this thread's two pixels
        Moments m[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) m[q] = Moments{make_float2(0.0f, 0.0f), make_float2(0.0f, 0.0f), 0.0f};
#pragma unroll
        for (int i = 0; i < kTaps + 1; ++i) {
            const float2 xy = h_xy[py + i][px], xx = h_xx[py + i][px];
            const float c = h_c[py + i][px];
#pragma unroll
            for (int q = 0; q < 2; ++q)
                if (i >= q && i - q < kTaps) add(m[q], tap(i - q), xy, xx, c);
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const float mx = m[q].xy.x, my = m[q].xy.y;
            const float vx = m[q].xx.x - mx * mx, vy = m[q].xx.y - my * my, cxy = m[q].c - mx * my;
            const float c1 = 0.01f * 0.01f, c2 = 0.03f * 0.03f;
            ss[q] += ((2.0f * mx * my + c1) * (2.0f * cxy + c2)) / ((mx * mx + my * my + c1) * (vx + vy + c2));
            const float2 v = s[ch][py + q + kHalo][px + kHalo];
            const float d = v.x - v.y;
            se[q] = fmaf(d, d, se[q]);
        }
        __syncthreads();  // the window sums are read before the next channel's
    }
    int reg[2] = {-1, -1};
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        ss[q] *= 1.0f / 3.0f;
        if (gx < w && gy + q < h) {
            reg[q] = regions ? (int)regions[(int64_t)(gy + q) * w + gx] : 0;
            if (reg[q] >= nreg) reg[q] = -1;
        }
    }
    // block sums per region
    for (int r = 0; r < nreg; ++r) {
        float a = (reg[0] == r ? se[0] : 0.0f) + (reg[1] == r ? se[1] : 0.0f);
        float b = (reg[0] == r ? ss[0] : 0.0f) + (reg[1] == r ? ss[1] : 0.0f);
        float c = (reg[0] == r ? 1.0f : 0.0f) + (reg[1] == r ? 1.0f : 0.0f);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a += __shfl_xor_sync(0xffffffffu, a, o);
            b += __shfl_xor_sync(0xffffffffu, b, o);
            c += __shfl_xor_sync(0xffffffffu, c, o);
        }
        if (lane == 0) {
            red[warp][r][0] = a;
            red[warp][r][1] = b;
            red[warp][r][2] = c;
        }
    }
    __syncthreads();
    if (tid < 3 * nreg) {
        const int r = tid / 3, q = tid - 3 * r;
        double t = 0.0;
        for (int v = 0; v < kMThreads / 32; ++v) t += (double)red[v][r][q];
        if (t != 0.0) atomicAdd(&acc[3 * r + q], t);
    }
}

}  // namespace

cudaError_t launch_image_metrics(const float *pred, const float *gt, int width, int height, const uint8_t *regions,
                                 int n_regions, double *acc, cudaStream_t s) {
    if (n_regions < 1 || n_regions > kMaxRegions) return cudaErrorInvalidValue;
    cudaError_t e = cudaMemsetAsync(acc, 0, sizeof(double) * 3 * n_regions, s);
    if (e != cudaSuccess || width == 0 || height == 0) return e;
    launch_k(k_image_metrics, dim3((unsigned)((width + kMW - 1) / kMW), (unsigned)((height + kMH - 1) / kMH)),
             dim3(kMThreads), 0, s, pred, gt, width, height, regions, n_regions, acc);
    return cudaGetLastError();
}

}  // namespace geer
