// train.cu -- the optimiser step of the training loop (Algorithm 2 with the
// 3DGS optimiser and parameterisation): one Adam step (Kingma and Ba) over the
// raw parameters mean, log-scale, quaternion, logit-opacity and SH, each group
// with its learning rate (SH degree 0 and the higher degrees apart). The
// renderer's gradients are with respect to the activated scale = exp(log-scale)
// and opacity = sigmoid(logit); the chain rule is applied here, and the
// activated values of the updated parameters are written for the next render.
//
// The moments m, v are flat over the groups [mean 3n | log-scale 3n | quat 4n |
// logit n | sh 3Kn] (K = (deg + 1)^2). A block takes 1024 elements of one group, four a
// thread, a block's width apart: every access coalesced whatever the group's alignment
// in the flat moments, all loads in flight before the first use (elementwise,
// HBM-bound: 16 B read and 12-16 B written per element).
#include <cmath>

#include "geer_internal.cuh"

namespace geer {
namespace {

struct AdamConst {
    float lr[6];  // mean, log-scale, quat, logit-opacity, SH degree 0, SH higher degrees
    float b1, b2, eps, inv_bc1, inv_bc2;  // inv_bc: 1 / (1 - beta^t)
};

enum : int { kGroupMean, kGroupScale, kGroupQuat, kGroupOpacity, kGroupSh, kGroups };

// One parameter group: values, gradients, the activated output (or null), its first
// element in the flat moments, its elements and its first block.
struct AdamGroup {
    float *p;
    const float *g;
    float *out;
    int64_t e0, count, block0;
};
struct AdamGroups {
    AdamGroup g[kGroups];
};

constexpr int kAdamThreads = 256, kAdamItems = 4, kAdamChunk = kAdamThreads * kAdamItems;

// (1,093,217 Gaussians of SH degree 3, 64.5M elements: 258 us, where one element a thread
// with the group and the SH position looked up per element took 528; four neighbouring
// elements a thread with 128-bit accesses, possible for n % 4 == 0 only: 259. With two elements a thread 277, with eight 263.)
__global__ void __launch_bounds__(kAdamThreads) k_adam_gaussians(AdamConst hp, AdamGroups gs, int K3,
                                                                 float *__restrict__ m, float *__restrict__ v) {
    grid_dep_sync();
    int group = 0;
    while (group + 1 < kGroups && (int64_t)blockIdx.x >= gs.g[group + 1].block0) ++group;
    const AdamGroup &G = gs.g[group];
    const int64_t off0 = ((int64_t)blockIdx.x - G.block0) * kAdamChunk;
    const int left = (int)min((int64_t)kAdamChunk, G.count - off0);
    float *__restrict__ p = G.p + off0;
    const float *__restrict__ gp = G.g + off0;
    float *__restrict__ mp = m + G.e0 + off0, *__restrict__ vp = v + G.e0 + off0;
    float x[kAdamItems], g[kAdamItems], mm[kAdamItems], vv[kAdamItems];
#pragma unroll
    for (int k = 0; k < kAdamItems; ++k) {
        const int i = k * kAdamThreads + threadIdx.x;
        if (i < left) {
            x[k] = p[i];
            g[k] = gp[i];
            mm[k] = mp[i];
            vv[k] = vp[i];
        }
    }
    // the chunk's first position in its Gaussian's SH row (block-uniform)
    const uint32_t row0 = group == kGroupSh ? (uint32_t)((uint64_t)off0 % (uint32_t)K3) : 0u;
#pragma unroll
    for (int k = 0; k < kAdamItems; ++k) {
        const int i = k * kAdamThreads + threadIdx.x;
        if (i >= left) break;
        float lr = hp.lr[group];
        if (group == kGroupSh && (row0 + (uint32_t)i) % (uint32_t)K3 >= 3u) lr = hp.lr[kGroups];
        float gi = g[k];
        if (group == kGroupScale) {
            gi *= expf(x[k]);  // d scale / d log-scale = scale
        } else if (group == kGroupOpacity) {
            const float s = 1.0f / (1.0f + expf(-x[k]));
            gi *= s * (1.0f - s);  // d sigmoid / d logit
        }
        const float m1 = hp.b1 * mm[k] + (1.0f - hp.b1) * gi;
        const float v1 = hp.b2 * vv[k] + (1.0f - hp.b2) * gi * gi;
        const float xn = x[k] - lr * (m1 * hp.inv_bc1) / (sqrtf(v1 * hp.inv_bc2) + hp.eps);
        p[i] = xn;
        mp[i] = m1;
        vp[i] = v1;
        if (G.out && group == kGroupScale) G.out[off0 + i] = expf(xn);
        if (G.out && group == kGroupOpacity) G.out[off0 + i] = 1.0f / (1.0f + expf(-xn));
    }
}

}  // namespace

cudaError_t launch_adam_gaussians(const geer_adam *hp, int64_t n, int32_t sh_degree, float *mean, float *log_scale,
                                  float *quat, float *logit_opacity, float *sh, const float *d_mean,
                                  const float *d_scale, const float *d_quat, const float *d_opacity,
                                  const float *d_sh, float *m, float *v, float *scale, float *opacity,
                                  cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    AdamConst c;
    c.lr[0] = hp->lr_mean;
    c.lr[1] = hp->lr_scale;
    c.lr[2] = hp->lr_quat;
    c.lr[3] = hp->lr_opacity;
    c.lr[4] = hp->lr_sh_dc;
    c.lr[5] = hp->lr_sh_rest;
    c.b1 = hp->beta1;
    c.b2 = hp->beta2;
    c.eps = hp->eps;
    c.inv_bc1 = (float)(1.0 / (1.0 - std::pow((double)hp->beta1, (double)hp->step)));
    c.inv_bc2 = (float)(1.0 / (1.0 - std::pow((double)hp->beta2, (double)hp->step)));
    const int K3 = 3 * (sh_degree + 1) * (sh_degree + 1);
    AdamGroups gs = {{{mean, d_mean, nullptr, 0, 3 * n, 0},
                             {log_scale, d_scale, scale, 3 * n, 3 * n, 0},
                             {quat, d_quat, nullptr, 6 * n, 4 * n, 0},
                             {logit_opacity, d_opacity, opacity, 10 * n, n, 0},
                             {sh, d_sh, nullptr, 11 * n, K3 * n, 0}}};
    int64_t blocks = 0;
    for (AdamGroup &g : gs.g) {
        g.block0 = blocks;
        blocks += (g.count + kAdamChunk - 1) / kAdamChunk;
    }
    if (blocks > 0x7fffffffll) return cudaErrorInvalidValue;
    launch_k(k_adam_gaussians, dim3((unsigned)blocks), dim3(kAdamThreads), 0, s, c, gs, K3, m, v);
    return cudaGetLastError();
}

}  // namespace geer
