// render.cu -- the per-ray render (Algorithm 1 per-CSF loop: Cano_Ray, Dist,
// BlendInOrder) and its backward (App. C, RenderCUDA stage).
//
// A BEAP tile (a camera sub-frustum) of 16 x 16 rays is processed by one block,
// one thread per ray, tiles taken in the order of descending pair count (the
// costliest first). A warp holds the 8 x 4 rays of one sub-tile (each half-warp
// 4 x 4 of them). The forward builds the tile's depth-ordered list on the fly
// from its super-tile's list (association test per entry), stages the records
// through shared memory in batches of BATCH, tests each entry once per sub-tile
// with a conservative bound (cull_keep) and every ray walks its sub-tile's
// entries front to back with the closed-form ray integral (Sec. 3.1):
//   d_u = W d, m_u = o_u x d_u, kappa = |m_u|^2 / |d_u|^2,
//   alpha = min(alpha_max, sigma exp(-kappa / 2)),
// skipping alpha < alpha_min and Gaussians whose closest approach lies behind
// the camera (o_u . d_u >= 0), stopping before the contributor that would take
// the transmittance below T_min (App. B.1 colour equation, 3DGS thresholds).
#include <algorithm>
#include <type_traits>

#include "geer_internal.cuh"

namespace geer {
namespace {

#ifndef GEER_FWD_MINB
#define GEER_FWD_MINB 4  // resident forward blocks per SM the registers must allow
#endif
#ifndef GEER_BWD_MINB
#define GEER_BWD_MINB 4
#endif
constexpr int kBatch = 256;    // list entries staged per batch (one per thread)
constexpr int kFwdUnroll = 4;  // list entries evaluated together
constexpr int kScan = 4;       // super-list loads in flight per thread in a list fill
constexpr float kNegHalfLog2e = -0.72134752044448170f;  // -log2(e) / 2

// A load of data written earlier in the same launch (CG: through L2, never a
// stale L1 line) or an ordinary one.
template <bool CG, typename T>
__device__ __forceinline__ T ld_cg(const T *p) {
    if constexpr (CG) return __ldcg(p);
    else return *p;
}

// 2^x by ex2.approx.ftz (error bound in the PTX manual): results below 2^-126 are 0. A
// hit's exponent argument is log2(alpha_min) or more, so that no alpha is lost down to
// alpha_min = 2^-126. (With exp2f the 1M-Gaussian training step takes 862 us in
// place of 846.)
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// 1/x by rcp.approx.ftz (error bound in the PTX manual), for x and 1/x that are normal
// numbers: |d_u|^2 at scales from 2^-60 to 2^60, and 1 - alpha. (With __fdividef(1, x) as well 882 us.)
__device__ __forceinline__ float rcp(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ int find_cam(const DevCam *cams, int ncams, int t) {
    int c = 0;
    for (int i = 1; i < ncams; ++i)
        if (cams[i].tile_base <= t) c = i;
    return c;
}

// One ray-Gaussian evaluation in the camera frame (Sec. 3.1): d_u = W d,
// m_u = o_u x d_u, kappa = |m_u|^2 / |d_u|^2 and the exponent argument
// log2(sigma) - kappa log2(e) / 2. The forward and the backward share it so that
// both take the same FP32 decisions.
struct Eval {
    float du0, du1, du2, m0, m1, m2, inv_dd, od, kappa, arg;
    bool hit;  // alpha >= alpha_min and the closest approach lies in front of the camera
};

__device__ __forceinline__ Eval evaluate(const float4 &a, const float4 &b, const float4 &c, const float4 &e, float dx,
                                         float dy, float dz, float log2_amin) {
    Eval v;
    v.du0 = a.x * dx + a.y * dy + a.z * dz;
    v.du1 = a.w * dx + b.x * dy + b.y * dz;
    v.du2 = b.z * dx + b.w * dy + c.x * dz;
    v.m0 = c.z * v.du2 - c.w * v.du1;
    v.m1 = c.w * v.du0 - c.y * v.du2;
    v.m2 = c.y * v.du1 - c.z * v.du0;
    const float mm = v.m0 * v.m0 + v.m1 * v.m1 + v.m2 * v.m2;
    v.inv_dd = rcp(v.du0 * v.du0 + v.du1 * v.du1 + v.du2 * v.du2);
    v.od = c.y * v.du0 + c.z * v.du1 + c.w * v.du2;
    v.kappa = mm * v.inv_dd;
    v.arg = fmaf(v.kappa, kNegHalfLog2e, e.x);
    v.hit = !(v.arg < log2_amin || v.od >= 0.0f);
    return v;
}

// The splat alpha (GEER_ALPHA_SPLAT, the local-affine model of EWA): the record
// holds the mean's screen angles and the conic (a = theta, phi, A, B; b.x = C);
// (ts, ps) are the ray's screen angles (atan2(x, z), atan2(y, z)). The exponent
// argument is log2(sigma) - D^T conic D log2(e) / 2 with D wrapped into
// [-pi, pi]. Sets arg and hit, and for the backward du0, du1 = D and kappa = q.
__device__ __forceinline__ Eval evaluate_splat(const float4 &a, const float4 &b, const float4 &e, float ts, float ps,
                                               float log2_amin) {
    constexpr float kTwoPi = 6.28318530717959f, kInvTwoPi = 0.159154943091895f;
    float dt = ts - a.x, dp = ps - a.y;
    dt = fmaf(-kTwoPi, rintf(dt * kInvTwoPi), dt);
    dp = fmaf(-kTwoPi, rintf(dp * kInvTwoPi), dp);
    Eval v{};
    const float q = fmaf(a.z * dt, dt, fmaf(2.0f * a.w * dt, dp, b.x * dp * dp));
    v.du0 = dt;
    v.du1 = dp;
    v.kappa = q;
    v.arg = fmaf(q, kNegHalfLog2e, e.x);
    v.hit = !(v.arg < log2_amin);
    return v;
}

__device__ __forceinline__ uint32_t lanemask_lt() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// A tile's super-tile list and its bit in the entries' masks.
struct TileList {
    const uint32_t *vals;  // item ids
    const uint32_t *mask;  // the mask word that holds the tile's bit, `words` apart
    const uint32_t *any;   // the same word of the groups' masks (32 entries each, aligned), `words` apart
    int words, shift;
    uint2 sr;              // [begin, end)
};

struct FillSmem {
    uint32_t wcnt[2][kScan * kTileWarps];  // a step writes one set while the slowest warp still reads the other
    uint32_t cut, taken;
    uint8_t grp[32];
};

constexpr uint32_t kChunk = 256;                // super-list entries that a fill takes or leaves together
constexpr uint32_t kLook = 31 * kChunk;         // entries of a step that skips empty groups of 32
constexpr uint32_t kSparse = 4;                 // tile entries of a step at or below which the next ones skip

// Inclusive (incl) and exclusive prefix of a step's 32 counts, one per lane.
__device__ __forceinline__ uint32_t scan_counts(const uint32_t *wcnt, uint32_t &incl) {
    const int lane = threadIdx.x & 31;
    const uint32_t c = wcnt[lane];
    incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    return incl - c;
}

// A tile's list is its super-tile's depth-ordered list filtered by its mask bit:
// appends the entries of [pos, end) that pass, in chunks of 256 super-list entries
// counted from the list's start, until s_id holds at least `want` entries or the
// list ends (so that s_id never takes more than want - 1 + 256; the chunks set the
// batches and with them the checkpoints' places). Each step loads kScan x 256
// entries at once (independent loads: the scan is bound by their latency); chunks it
// did not take are read again by the next call. After a step with hardly an entry
// of the tile, a step looks at the or'd masks of 248 groups of 32 entries and reads
// those of at most 32 groups that hold one (the serving scene's sparsest tiles own
// 1 entry in 400 of an 800K-entry list: 1.1 ms of a batch's 2.9 were one such
// block's scan). Block-uniform (pos, sparse, want and s_cnt are the same in every
// thread); s_id is visible on return.
__device__ __forceinline__ void fill_list(const TileList &tl, uint32_t &pos, bool &sparse, int want, uint32_t *s_id,
                                          uint32_t *s_pos, int &s_cnt, FillSmem &sf) {
    constexpr int kWarps = kTileWarps;
    static_assert(kScan * kWarps == 32 && kChunk == kTilePix, "a warp scans a step's counts with a lane each");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t end = tl.sr.y;
    if (s_cnt >= want || pos >= end) return;
    for (int par = 0; s_cnt < want && pos < end; par ^= 1) {
        uint32_t id[kScan], at[kScan], bal[kScan], incl;
        if (!sparse) {
#pragma unroll
            for (int r = 0; r < kScan; ++r) {
                at[r] = pos + (uint32_t)r * kChunk + threadIdx.x;
                bal[r] = at[r] < end ? tl.mask[(size_t)at[r] * tl.words] : 0u;
                id[r] = at[r] < end ? tl.vals[at[r]] : 0u;
            }
#pragma unroll
            for (int r = 0; r < kScan; ++r) {
                bal[r] = __ballot_sync(0xffffffffu, bal[r] >> tl.shift & 1u);
                if (lane == 0) sf.wcnt[par][r * kWarps + warp] = __popc(bal[r]);
            }
            __syncthreads();
            const uint32_t excl = scan_counts(sf.wcnt[par], incl);
            uint32_t taken = 0;
            sparse = __shfl_sync(0xffffffffu, incl, 31) <= kSparse;
#pragma unroll
            for (int r = 0; r < kScan; ++r) {
                const uint32_t base = __shfl_sync(0xffffffffu, excl, r * kWarps + warp);
                const uint32_t upto = __shfl_sync(0xffffffffu, incl, r * kWarps + kWarps - 1);
                if (s_cnt + (int)taken >= want) break;  // block-uniform: every warp scans the same counts
                if (bal[r] >> lane & 1u) {
                    const int k = s_cnt + (int)(base + __popc(bal[r] & lanemask_lt()));
                    s_id[k] = id[r];
                    if (s_pos) s_pos[k] = at[r];
                }
                taken = upto;
                pos += kChunk;
            }
            s_cnt += (int)taken;
            continue;
        }
        // the groups of [pos, pos + kLook) that hold an entry of the tile
        const uint32_t g0 = pos >> 5, lim = min(pos + kLook, end);
        const uint32_t g = g0 + threadIdx.x;
        const bool any = (g << 5) < lim && (tl.any[(size_t)g * tl.words] >> tl.shift & 1u);
        const uint32_t b = __ballot_sync(0xffffffffu, any);
        if (lane == 0) sf.wcnt[par][warp] = __popc(b);
        if (threadIdx.x == 0) sf.taken = 0u;
        __syncthreads();
        uint32_t pre = 0, n = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const uint32_t c = sf.wcnt[par][w];
            pre += w < warp ? c : 0u;
            n += c;
        }
        if (n > 32u) {  // dense again
            sparse = false;
            continue;
        }
        if (any) sf.grp[pre + __popc(b & lanemask_lt())] = (uint8_t)threadIdx.x;
        par ^= 1;
        __syncthreads();
        const uint32_t gs = (uint32_t)lane < n ? (g0 + sf.grp[lane]) << 5 : 0xffffffffu;
#pragma unroll
        for (int r = 0; r < kScan; ++r) {
            const uint32_t first = __shfl_sync(0xffffffffu, gs, r * kWarps + warp);
            at[r] = first + (uint32_t)lane;
            const bool in = first != 0xffffffffu && at[r] >= pos && at[r] < lim;
            bal[r] = in ? tl.mask[(size_t)at[r] * tl.words] : 0u;
            id[r] = in ? tl.vals[at[r]] : 0u;
        }
#pragma unroll
        for (int r = 0; r < kScan; ++r) {
            bal[r] = __ballot_sync(0xffffffffu, bal[r] >> tl.shift & 1u);
            if (lane == 0) sf.wcnt[par][r * kWarps + warp] = __popc(bal[r]);
        }
        __syncthreads();
        const uint32_t excl = scan_counts(sf.wcnt[par], incl);
        const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
        uint32_t rank[kScan], stop = lim;
#pragma unroll
        for (int r = 0; r < kScan; ++r)
            rank[r] = __shfl_sync(0xffffffffu, excl, r * kWarps + warp) + __popc(bal[r] & lanemask_lt());
        const bool cuts = s_cnt + (int)total >= want;
        if (cuts) {  // the chunk of entry number `want` is the last one to take
#pragma unroll
            for (int r = 0; r < kScan; ++r)
                if ((bal[r] >> lane & 1u) && rank[r] == (uint32_t)(want - s_cnt) - 1u) sf.cut = (at[r] - pos) / kChunk;
            __syncthreads();
            stop = pos + (sf.cut + 1u) * kChunk;
        }
#pragma unroll
        for (int r = 0; r < kScan; ++r) {
            const bool take = (bal[r] >> lane & 1u) && at[r] < stop;
            if (take) {
                s_id[s_cnt + (int)rank[r]] = id[r];
                if (s_pos) s_pos[s_cnt + (int)rank[r]] = at[r];
            }
            if (cuts) {  // how many that is
                const uint32_t most = __reduce_max_sync(0xffffffffu, take ? rank[r] + 1u : 0u);
                if (lane == 0 && most) atomicMax(&sf.taken, most);
            }
        }
        if (cuts) __syncthreads();
        s_cnt += cuts ? (int)sf.taken : (int)total;
        pos = cuts ? stop : pos + kLook;
    }
    __syncthreads();
}

// Moves the s_cnt - cnt entries not yet consumed (fewer than 256) to the front.
__device__ __forceinline__ void shift_list(uint32_t *s_id, uint32_t *s_pos, int cnt, int &s_cnt) {
    const int rem = s_cnt - cnt;
    uint32_t keep = 0, keep_pos = 0;
    if ((int)threadIdx.x < rem) {
        keep = s_id[cnt + threadIdx.x];
        if (s_pos) keep_pos = s_pos[cnt + threadIdx.x];
    }
    __syncthreads();
    if ((int)threadIdx.x < rem) {
        s_id[threadIdx.x] = keep;
        if (s_pos) s_pos[threadIdx.x] = keep_pos;
    }
    s_cnt = rem;
}

// The same filter walking the super-tile list backwards: appends the passing
// entries of [beg, pos) in descending position order (the tile list read back to
// front) until s_id holds at least kBatch entries or pos reaches beg.
__device__ __forceinline__ void fill_list_rev(const TileList &tl, uint32_t &pos, uint32_t beg, uint32_t *s_id,
                                              int &s_cnt, uint32_t *s_wcnt) {
    constexpr int kThreads = kTilePix;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    while (s_cnt < kBatch && pos > beg) {
        bool ok = false;
        uint32_t id = 0;
        if (pos - beg > threadIdx.x) {
            const uint32_t i = pos - 1 - threadIdx.x;
            ok = tl.mask[(size_t)i * tl.words] >> tl.shift & 1u;
            if (ok) id = tl.vals[i];
        }
        const uint32_t bal = __ballot_sync(0xffffffffu, ok);
        if (lane == 0) s_wcnt[warp] = __popc(bal);
        __syncthreads();
        uint32_t base = 0, tot = 0;
#pragma unroll
        for (int w = 0; w < kThreads / 32; ++w) {
            const uint32_t c = s_wcnt[w];
            base += w < warp ? c : 0u;
            tot += c;
        }
        if (ok) s_id[s_cnt + base + __popc(bal & lanemask_lt())] = id;
        __syncthreads();
        s_cnt += (int)tot;
        pos = pos - beg > (uint32_t)kThreads ? pos - kThreads : beg;
    }
}

// Shared-memory working set of one block's walk over its tile's list.
struct WalkSmem {
    float4 rec[(kBatch + 1) * 4];       // records of the current batch; forward: the last one is never hit
    uint32_t id[kBatch + kTilePix];     // tile-list entries found by the filter (item ids)
    uint2 hit[kBatch];                  // per entry: one byte per backward warp (16 x 2 rays), nonzero if a ray hit it
    union {
        struct {                        // forward
            uint32_t pos[kBatch + kTilePix];    // the entries' positions in the super-tile list
            float4 conic[kBatch * 2];           // the batch's quadratics
            uint16_t list[kTileWarps][kBatch + kFwdUnroll];  // each sub-tile's entries of the batch (byte offsets in rec)
            float4 sub[kTileWarps];             // the sub-tiles' rectangles (centre, half sizes) in the tile's chart
            float2 ray[kTileWarps][32];         // their rays' points there
            float4 frame[3];                    // the chart's axes c, e1, e2 (splat: the reference angles)
            uint32_t ext[2];                    // the largest |x|, |y| of the tile's rays (FP32 bits)
        };
        struct {                        // backward
            float acc[kBatch][17];              // the batch's sums over the tile's rays
            uint8_t blist[kTileWarps][kBatch];  // each warp's entries of the batch
            uint32_t odd;                       // a staged colour takes warp_sum's ODD sums from here on
        };
    };
    FillSmem fill;
    uint32_t maxlast, walkpos;       // the tile's last contributor and its super-list position + 1
    uint32_t nck, next_ck;           // forward: checkpoints recorded, list index of the next one
    uint32_t wacc[kTilePix];         // forward: each thread's count of backward steps
    uint32_t ckw[kCkptMax];          // forward: the counts at the checkpoints (work: then the walk's)
    uint32_t ckB[kCkptMax];          // forward: the checkpoints' tile-list indices
    uint32_t work, pend;             // forward: a checkpoint's count of backward steps; its index + 1 while due
    int cam;
};

// Item `id`'s 64-byte record (4 x 16 B). An id beyond the items (a guard failure)
// gives a record that no ray hits: W = 0 gives kappa = 0/0 and o_u . d_u = 0 (the
// exact integral's test fails), and log2(sigma) = -inf fails the splat alpha's.
__device__ __forceinline__ void load_record(float4 q[4], const Record *__restrict__ rec, uint32_t id, uint64_t items,
                                            uint32_t site, uint32_t *misc) {
    if (in_bounds(id, items, site, misc)) {
        const float4 *src = reinterpret_cast<const float4 *>(rec + id);
#pragma unroll
        for (int k = 0; k < 4; ++k) q[k] = src[k];
    } else {
        q[0] = q[1] = q[2] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        q[3] = make_float4(-INFINITY, 0.0f, 0.0f, 0.0f);
    }
}

// ---- Sub-tile culling -------------------------------------------------------
// A ray hits an entry where kappa = |o_u x W d|^2 / |W d|^2 <= kappa_max =
// 2 ln(sigma / alpha_min). kappa does not depend on d's length: with d scaled to
// c + x e1 + y e2 (the tile's chart: c its central direction, e1 and e2 orthonormal
// to it) that is Q(x, y) = |o_u x W d|^2 - kappa_max |W d|^2 <= 0, a quadratic in
// (x, y). No ray of a sub-tile hits the entry when a lower bound of Q over the
// rectangle of its rays' points is positive: the tangent plane's least value
// (valid for a convex Q) at the rectangle's point nearest the conic's centre, or,
// when Q is not convex, at the rectangle's centre with the curvature subtracted.
// A conic that covers only a few rays' share of the rectangle is also evaluated
// at all 32 rays.
//
// A thread computes one entry's quadratic (~130 instructions), each warp then tests
// 32 entries at a time against its sub-tile, a lane per entry (~35 instructions,
// ~210 more for the rays), where evaluating one entry costs a warp ~50 whether or
// not a ray of it hits. Of the 1M-Gaussian fisheye scene's (entry, sub-tile) pairs
// 28% have a ray that hits and 38% pass the test, of the 500k shell's 17% and 23%
// (36% without the rays; 70% in the corner tiles that end its launch, 9% with
// them). us a pass with the tile masks of the lists, before and after: 500k shell
// at 1024 x 1024 305 -> 262, 4096 Gaussians at 128 x 128 131 -> 118.5.
//
// The test never drops what evaluate() / evaluate_splat() calls a hit: e bounds
// the FP32 errors of both sides. evaluate(): W d carries 4 ulp of |W| |d|, which
// o_u x multiplies by |o_u|; kappa, its exponent argument and the quotient a few
// ulp each (in kappa_max's margin); the chart point 8 ulp of the direction. Q: 67
// ulp of the squared magnitudes it is built from. Entries of extreme scale (where
// the quotient under- or overflows) are always kept.
struct Conic {
    float q0, gx, gy, a, b, c;  // Q(x, y) = q0 + 2 gx x + 2 gy y + a x^2 + 2 b x y + c y^2
    float e;                    // error bound: out where the lower bound exceeds e
};

template <bool SPLAT>
__device__ __forceinline__ Conic cull_conic(const float4 q[4], const float4 *frame, const uint32_t *ext,
                                            float log2_amin) {
    Conic v;
    const float hx = __uint_as_float(ext[0]), hy = __uint_as_float(ext[1]);
    // kappa_max, with the rounding of the hit test's exponent argument in it
    const float km = fmaf(fmaxf(q[3].x - log2_amin, 0.0f), 1.38632f, 2e-5f);
    if (SPLAT) {
        constexpr float kTwoPi = 6.28318530717959f, kInvTwoPi = 0.159154943091895f;
        float dt = frame[0].x - q[0].x, dp = frame[0].y - q[0].y;
        dt = fmaf(-kTwoPi, rintf(dt * kInvTwoPi), dt);
        dp = fmaf(-kTwoPi, rintf(dp * kInvTwoPi), dp);
        v.a = q[0].z;
        v.b = q[0].w;
        v.c = q[1].x;
        v.gx = fmaf(v.a, dt, v.b * dp);
        v.gy = fmaf(v.b, dt, v.c * dp);
        v.q0 = fmaf(v.gx, dt, v.gy * dp) - km;
        const float s = fabsf(dt) + hx, t = fabsf(dp) + hy, ab = fabsf(v.b);
        const float as = fmaf(v.a, s, ab * t), ct = fmaf(v.c, t, ab * s);
        v.e = 8e-6f * fmaf(as, s, ct * t) + 8e-6f * (as + ct) + 1e-10f * (v.a + v.c + 2.0f * ab);
        if (!(s < 3.14f && t < 3.14f)) v.e = INFINITY;  // a wrap of the difference inside the tile: kept
        return v;
    }
    const float4 &A = q[0], &B = q[1], &C = q[2];  // W00 W01 W02 W10 | W11 W12 W20 W21 | W22 ou0 ou1 ou2
    const float ox = C.y, oy = C.z, oz = C.w;
    const float4 f0 = frame[0], f1 = frame[1], f2 = frame[2];
    const auto row0 = [&](const float4 &f) { return fmaf(A.x, f.x, fmaf(A.y, f.y, A.z * f.z)); };
    const auto row1 = [&](const float4 &f) { return fmaf(A.w, f.x, fmaf(B.x, f.y, B.y * f.z)); };
    const auto row2 = [&](const float4 &f) { return fmaf(B.z, f.x, fmaf(B.w, f.y, C.x * f.z)); };
    const float u0 = row0(f0), u1 = row1(f0), u2 = row2(f0);  // W d at the chart's origin
    const float v0 = row0(f1), v1 = row1(f1), v2 = row2(f1);  // and its x
    const float w0 = row0(f2), w1 = row1(f2), w2 = row2(f2);  // and y derivatives
    const float m0 = oy * u2 - oz * u1, m1 = oz * u0 - ox * u2, m2 = ox * u1 - oy * u0;  // the same of o_u x W d
    const float k0 = oy * v2 - oz * v1, k1 = oz * v0 - ox * v2, k2 = ox * v1 - oy * v0;
    const float l0 = oy * w2 - oz * w1, l1 = oz * w0 - ox * w2, l2 = ox * w1 - oy * w0;
    const float mm = m0 * m0 + m1 * m1 + m2 * m2, kk = k0 * k0 + k1 * k1 + k2 * k2, ll = l0 * l0 + l1 * l1 + l2 * l2;
    v.q0 = fmaf(-km, u0 * u0 + u1 * u1 + u2 * u2, mm);
    v.gx = fmaf(-km, u0 * v0 + u1 * v1 + u2 * v2, m0 * k0 + m1 * k1 + m2 * k2);
    v.gy = fmaf(-km, u0 * w0 + u1 * w1 + u2 * w2, m0 * l0 + m1 * l1 + m2 * l2);
    v.a = fmaf(-km, v0 * v0 + v1 * v1 + v2 * v2, kk);
    v.b = fmaf(-km, v0 * w0 + v1 * w1 + v2 * w2, k0 * l0 + k1 * l1 + k2 * l2);
    v.c = fmaf(-km, w0 * w0 + w1 * w1 + w2 * w2, ll);
    // the errors, from |W| |d| (n), |o_u| and the largest |m| of the tile (bm)
    const float r0 = A.x * A.x + A.y * A.y + A.z * A.z, r1 = A.w * A.w + B.x * B.x + B.y * B.y,
                r2 = B.z * B.z + B.w * B.w + C.x * C.x;
    const float sk = sqrtf(km), n = sqrtf((r0 + r1 + r2) * fmaf(hx, hx, fmaf(hy, hy, 1.001f)));
    const float on = sqrtf(ox * ox + oy * oy + oz * oz), bm = sqrtf(mm) + hx * sqrtf(kk) + hy * sqrtf(ll);
    const float cc = 2e-6f * n * (on + sk);
    v.e = fmaf(cc, fmaf(2.0f * sk, n, cc), 4e-6f * fmaf(bm, fmaf(on, n, bm), km * n * n));
    if (!(n < 1e18f && fminf(r0, fminf(r1, r2)) > 1e-30f)) v.e = INFINITY;  // extreme scales: kept
    return v;
}

// Whether a ray in the rectangle r (centre x, y, half sizes) may hit the entry.
// few: the conic covers the share of about eight rays or less.
__device__ __forceinline__ bool cull_keep(const Conic &v, const float4 &r, bool &few) {
    const float det = fmaf(v.a, v.c, -v.b * v.b);
    const bool convex = v.a > 0.0f && v.c > 0.0f && det > 1e-6f * v.a * v.c;
    float x = r.x, y = r.y;
    few = false;
    if (convex) {  // the point of the rectangle nearest the conic's centre (any point serves)
        const float id = __fdividef(1.0f, det);
        const float cx = (v.b * v.gy - v.c * v.gx) * id, cy = (v.b * v.gx - v.a * v.gy) * id;
        x = fminf(fmaxf(cx, r.x - r.z), r.x + r.z);
        y = fminf(fmaxf(cy, r.y - r.w), r.y + r.w);
        // its area is pi w / sqrt(det), w = -Q at the centre, the rectangle's 4 r.z r.w
        const float w = -fmaf(v.gx, cx, fmaf(v.gy, cy, v.q0));
        few = w * w * id < 0.1f * r.z * r.z * r.w * r.w;
    }
    const float hx = fmaf(v.a, x, fmaf(v.b, y, v.gx)), hy = fmaf(v.b, x, fmaf(v.c, y, v.gy));  // half gradient
    // Q at (x, y) = q0 + (gx + hx) x + (gy + hy) y; the tangent plane's least value over the rectangle
    const float at = fmaf(v.gx + hx, x, fmaf(v.gy + hy, y, v.q0));
    float low = at + 2.0f * (fmaf(hx, r.x - x, hy * (r.y - y)) - fmaf(fabsf(hx), r.z, fabsf(hy) * r.w));
    if (!convex)
        low += fminf(v.a, 0.0f) * r.z * r.z + fminf(v.c, 0.0f) * r.w * r.w - 2.0f * fabsf(v.b) * r.z * r.w;
    return !(low > v.e);  // a NaN keeps the entry
}

// The least Q over the sub-tile's rays (a NaN where there is no ray).
__device__ __forceinline__ bool cull_keep_rays(const Conic &v, const float2 *ray) {
    float low = NAN;
#pragma unroll 8
    for (int k = 0; k < 32; k += 2) {
        const float4 r = *reinterpret_cast<const float4 *>(ray + k);
        low = fminf(low, fmaf(r.x, fmaf(v.a, r.x, fmaf(2.0f * v.b, r.y, 2.0f * v.gx)),
                              fmaf(r.y, fmaf(v.c, r.y, 2.0f * v.gy), v.q0)));
        low = fminf(low, fmaf(r.z, fmaf(v.a, r.z, fmaf(2.0f * v.b, r.w, 2.0f * v.gx)),
                              fmaf(r.w, fmaf(v.c, r.w, 2.0f * v.gy), v.q0)));
    }
    return !(low > v.e);
}
constexpr int kRaysFrom = 6;  // entries of 32 for which testing all rays is cheaper than evaluating them

// The tile's chart, its sub-tiles' rectangles and rays there (block-wide, ends in a
// barrier). c: the mean direction of the tile's rays; e1 and e2: the projection of
// the x axis (of the y axis for a c near the x axis) and the normal to it. The
// rectangles carry 8 ulp of rounding. A sub-tile with a ray more than ~84 degrees
// from c, or without rays, gets infinite half sizes (its low is -infinity or NaN:
// its test never drops an entry). Splat: the rays' screen angles about the first
// ray's.
template <bool SPLAT>
__device__ __forceinline__ void sub_tiles(WalkSmem &sm, bool inside, float dx, float dy, float dz) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float x, y;
    bool bad = false;
    if (threadIdx.x < 2) sm.ext[threadIdx.x] = 0u;
    if (SPLAT) {
        if (threadIdx.x == 0) sm.frame[0] = make_float4(dx, dy, 0.0f, 0.0f);  // the tile's first ray is in the image
        __syncthreads();
        x = dx - sm.frame[0].x;
        y = dy - sm.frame[0].y;
    } else {
        const float len = sqrtf(fmaf(dx, dx, fmaf(dy, dy, dz * dz))), inv = inside && len > 0.0f ? 1.0f / len : 0.0f;
        float s0 = dx * inv, s1 = dy * inv, s2 = dz * inv;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            s0 += __shfl_xor_sync(0xffffffffu, s0, o);
            s1 += __shfl_xor_sync(0xffffffffu, s1, o);
            s2 += __shfl_xor_sync(0xffffffffu, s2, o);
        }
        if (lane == 0) sm.sub[warp] = make_float4(s0, s1, s2, 0.0f);
        __syncthreads();
        if (warp == 0) {
            const float4 t = sm.sub[lane & (kTileWarps - 1)];
            float c0 = t.x, c1 = t.y, c2 = t.z;
#pragma unroll
            for (int o = kTileWarps / 2; o > 0; o >>= 1) {
                c0 += __shfl_xor_sync(0xffffffffu, c0, o);
                c1 += __shfl_xor_sync(0xffffffffu, c1, o);
                c2 += __shfl_xor_sync(0xffffffffu, c2, o);
            }
            const float ic = rsqrtf(fmaf(c0, c0, fmaf(c1, c1, c2 * c2)));
            c0 *= ic;
            c1 *= ic;
            c2 *= ic;
            // a e1 (or e2) = axis - c (c . axis), normalised; the other one by the cross product
            const bool ax = fabsf(c0) < 0.9f;
            const float p = ax ? c0 : c1;
            float a0 = fmaf(-c0, p, ax ? 1.0f : 0.0f), a1 = fmaf(-c1, p, ax ? 0.0f : 1.0f), a2 = -c2 * p;
            const float ia = rsqrtf(fmaf(a0, a0, fmaf(a1, a1, a2 * a2)));
            a0 *= ia;
            a1 *= ia;
            a2 *= ia;
            if (lane == 0) {
                sm.frame[0] = make_float4(c0, c1, c2, 0.0f);
                sm.frame[1] = make_float4(a0, a1, a2, 0.0f);
                sm.frame[2] = make_float4(c1 * a2 - c2 * a1, c2 * a0 - c0 * a2, c0 * a1 - c1 * a0, 0.0f);
            }
        }
        __syncthreads();
        const float4 c = sm.frame[0], e1 = sm.frame[1], e2 = sm.frame[2];
        const float dc = fmaf(dx, c.x, fmaf(dy, c.y, dz * c.z)), idc = 1.0f / dc;
        x = fmaf(dx, e1.x, fmaf(dy, e1.y, dz * e1.z)) * idc;
        y = fmaf(dx, e2.x, fmaf(dy, e2.y, dz * e2.z)) * idc;
        bad = !(dc > 0.1f * len);
    }
    const unsigned in = __ballot_sync(0xffffffffu, inside);
    const bool ok = in && !__any_sync(0xffffffffu, inside && bad);
    float x0 = inside ? x : INFINITY, x1 = inside ? x : -INFINITY, y0 = inside ? y : INFINITY, y1 = inside ? y : -INFINITY;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        x0 = fminf(x0, __shfl_xor_sync(0xffffffffu, x0, o));
        x1 = fmaxf(x1, __shfl_xor_sync(0xffffffffu, x1, o));
        y0 = fminf(y0, __shfl_xor_sync(0xffffffffu, y0, o));
        y1 = fmaxf(y1, __shfl_xor_sync(0xffffffffu, y1, o));
    }
    sm.ray[warp][lane] = ok && inside ? make_float2(x, y) : make_float2(NAN, NAN);
    if (lane == 0) {
        const float mx = fmaxf(fabsf(x0), fabsf(x1)), my = fmaxf(fabsf(y0), fabsf(y1));
        sm.sub[warp] = ok ? make_float4(0.5f * (x0 + x1), 0.5f * (y0 + y1), 0.5f * (x1 - x0) + (1e-6f * mx + 1e-7f),
                                        0.5f * (y1 - y0) + (1e-6f * my + 1e-7f))
                          : make_float4(0.0f, 0.0f, INFINITY, INFINITY);
        if (ok) {  // (an atomic max of non-negative FP32 bits)
            atomicMax(&sm.ext[0], __float_as_uint(mx * 1.00001f + 1e-6f));
            atomicMax(&sm.ext[1], __float_as_uint(my * 1.00001f + 1e-6f));
        }
    }
    __syncthreads();
}

// A tile's super-tile list range must lie within the sorted pairs; a guard
// failure leaves the tile an empty list.
__device__ __forceinline__ uint2 checked_range(uint2 sr, int64_t cap_pairs, uint32_t site, uint32_t *misc) {
    if (!in_bounds(sr.y, (uint64_t)cap_pairs + 1u, site, misc) || !in_bounds(sr.x, (uint64_t)sr.y + 1u, site, misc))
        return make_uint2(0u, 0u);
    return sr;
}

// A thread's ray in the forward: warp w holds sub-tile w's 8 x 4 rays (two columns
// of four sub-tiles). Compact warps meet fewer footprints than rows do: a disc of
// radius r pixels meets (8 + 2r)(4 + 2r) placements of an 8 x 4 warp,
// (16 + 2r)(2 + 2r) of a 16 x 2 one. The backward's warps hold 16 x 2 rays (ray =
// thread): the order of its sums, and with it the last digits of ill-conditioned
// gradients (needles close to a camera), stays what it is.
__device__ __forceinline__ int fwd_ray(int tid) {
    return ((tid >> 6) * 4 + ((tid >> 3) & 3)) * kTile + ((tid >> 5) & 1) * 8 + (tid & 7);
}

// Per-ray forward state (n_eval: entries evaluated, set when the walk ends).
struct FwdRay {
    float T, cr, cg, cb;
    uint32_t last, n_eval, n_applied;
    bool done;
};

// Composites the sub-tile's entries of the staged batch (list: n byte offsets of
// their records, padded to a multiple of kFwdUnroll with a record that no ray
// hits) into ray state f, front to back (App. B.1 colour equation), until the
// ray terminates: kFwdUnroll entries are evaluated together (independent work for
// the scheduler on long walks), then composited strictly in list order. Entry j
// of the batch has tile-list index n_list + j. hit_b: the hit byte of entry 0 of the
// ray's backward warp (8 bytes per entry).
template <bool SPLAT>
__device__ __forceinline__ void walk_entries(const float4 *srec, const uint16_t *list, int n, uint32_t n_list, uint32_t *misc,
                                             uint8_t *hit_b, const Params &p, float log2_amin, float dx, float dy,
                                             float dz, FwdRay &f) {
    static_assert(kFwdUnroll == 4, "four 16-bit offsets per shared load");
    for (int k = 0; k < n && !f.done; k += kFwdUnroll) {
        const uint2 o2 = *reinterpret_cast<const uint2 *>(list + k);
        uint32_t off[kFwdUnroll] = {o2.x & 0xffffu, o2.x >> 16, o2.y & 0xffffu, o2.y >> 16};
        const uint32_t drop = GEER_CHECKED ? (off[0] & 1u) | (off[1] & 1u) << 1 | (off[2] & 1u) << 2 | (off[3] & 1u) << 3 : 0u;
#pragma unroll
        for (int u = 0; u < kFwdUnroll; ++u) off[u] &= ~(GEER_CHECKED ? 1u : 0u);
        Eval v[kFwdUnroll];
        float4 e[kFwdUnroll];
#pragma unroll
        for (int u = 0; u < kFwdUnroll; ++u) {
            const float4 *r = reinterpret_cast<const float4 *>(reinterpret_cast<const char *>(srec) + off[u]);
            const float4 a = r[0];  // W00 W01 W02 W10
            const float4 b = r[1];  // W11 W12 W20 W21
            const float4 c = r[2];  // W22 ou0 ou1 ou2
            e[u] = r[3];            // log2 sigma, r, g, b
            v[u] = SPLAT ? evaluate_splat(a, b, e[u], dx, dy, log2_amin) : evaluate(a, b, c, e[u], dx, dy, dz, log2_amin);
        }
        // after the group's record loads (a byte store may alias them); the
        // same value from every lane: no race
#pragma unroll
        for (int u = 0; u < kFwdUnroll; ++u)
            if (v[u].hit) hit_b[off[u] >> 3] = 1;
        // branch-free per entry (predicated updates): with data-dependent branches
        // the four steps cost a reconvergence each
#pragma unroll
        for (int u = 0; u < kFwdUnroll; ++u) {
            const float alpha = fminf(ex2(v[u].arg), p.alpha_max);
            const float Tn = f.T * (1.0f - alpha);
            const uint32_t at = n_list + (off[u] >> 6) + 1u;
            const bool live = v[u].hit && !f.done;
            if (GEER_CHECKED && live && (drop >> u & 1u)) in_bounds(n_list + (off[u] >> 6), 0u, kSiteFwdCull, misc);
            if (live && Tn < p.T_min) {
                f.done = true;
                f.n_eval = at;  // entries up to this one
            }
            if (live && !(Tn < p.T_min)) {
                const float wgt = alpha * f.T;
                f.cr = fmaf(wgt, e[u].y, f.cr);
                f.cg = fmaf(wgt, e[u].z, f.cg);
                f.cb = fmaf(wgt, e[u].w, f.cb);
                f.T = Tn;
                ++f.n_applied;
                f.last = at;
            }
        }
    }
}

constexpr int kFewEntries = 8;  // tiles of up to this many entries are walked without bounds

// The tile's forward walk (the per-CSF loop of Algorithm 1): its list is the
// super-tile list [sr.x, sr.y) filtered by the association test; batches of
// records are staged in shared memory and each ray composites them front to
// back until it terminates. On return sm.maxlast / sm.walkpos hold the tile's
// walk record: [sr.x, walkpos) of the super-tile list holds tile-list entries
// 0 .. maxlast - 1.
// SPLAT: the splat alpha (GEER_ALPHA_SPLAT) in place of the ray integral;
// (dx, dy) then carry the ray's screen angles.
template <bool SPLAT>
__device__ __forceinline__ void forward_walk(WalkSmem &sm, const TileList &tl, const Record *__restrict__ rec,
                                             const Params &p, float dx, float dy, float dz,
                                             uint2 *__restrict__ hit_rec,
                                             uint32_t *__restrict__ id_rec, int64_t hit_entries, uint64_t items,
                                             uint32_t *misc,
                                             float4 *__restrict__ ckpt, uint2 *__restrict__ ckpt_at,
                                             FwdRay &f) {
    constexpr int kThreads = kTilePix;
    static_assert(kBatch == kThreads, "one record per thread and batch");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint8_t *const hit_b = reinterpret_cast<uint8_t *>(sm.hit) + fwd_ray(tid) / 32;  // the ray's byte of entry 0
    if (tid == 0) {
        sm.maxlast = 0u;
        sm.walkpos = tl.sr.x;
        sm.nck = 0u;
        sm.next_ck = ckpt ? kCkptFirst : 0xffffffffu;
        sm.work = 0u;
        sm.pend = 0u;
    }
    if (tid < 4) sm.rec[kBatch * 4 + tid] = make_float4(tid == 3 ? -INFINITY : 0.0f, 0.0f, 0.0f, 0.0f);
    sm.wacc[tid] = 0u;
    const float log2_amin = log2f(p.alpha_min);
    uint32_t pos = tl.sr.x, n_list = 0;
    bool sparse = false;
    int s_cnt = 0, want = 64;
    while (true) {
        if (__syncthreads_count(f.done) == kThreads) break;
        // batches grow 64, 128, ... kBatch: most rays of a dense scene stop early
        fill_list(tl, pos, sparse, want, sm.id, sm.pos, s_cnt, sm.fill);
        want = min(2 * want, kBatch);
        const int cnt = min(s_cnt, kBatch);
        if (cnt == 0) break;
        // a tile of a few entries walks them all: the bounds of its sub-tiles and entries
        // cost as much as ~10 entries (17K Gaussians on 1432 x 1377: 88 us with them
        // everywhere, 70 so; at 16 entries 72). It has no second batch: only a list's end cuts one short.
        const bool cull = n_list > 0 || cnt > kFewEntries;
        if (cull && n_list == 0) sub_tiles<SPLAT>(sm, !f.done, dx, dy, dz);
        if (tid < cnt) {  // entry tid: its record and quadratic
            float4 q[4];
            load_record(q, rec, sm.id[tid], items, kSiteFwdItem, misc);
#pragma unroll
            for (int k = 0; k < 4; ++k) sm.rec[tid * 4 + k] = q[k];
            if (cull) {
                const Conic v = cull_conic<SPLAT>(q, sm.frame, sm.ext, log2_amin);
                sm.conic[2 * tid] = make_float4(v.q0, v.gx, v.gy, v.a);
                sm.conic[2 * tid + 1] = make_float4(v.b, v.c, v.e, 0.0f);
            }
            sm.hit[tid] = make_uint2(0u, 0u);
        }
        __syncthreads();
        if (!__all_sync(0xffffffffu, f.done)) {
            // the entries this warp's rays may hit, in list order
            uint16_t *const list = sm.list[warp];
            const float4 rect = sm.sub[warp];
            int n = 0;
            for (int g = 0; g < cnt; g += 32) {
                bool keep = !cull && g + lane < cnt, few = false;
                Conic v{};
                if (cull && g + lane < cnt) {
                    const float4 u = sm.conic[2 * (g + lane)], w = sm.conic[2 * (g + lane) + 1];
                    v = Conic{u.x, u.y, u.z, u.w, w.x, w.y, w.z};
                    keep = cull_keep(v, rect, few);
                }
                if (__popc(__ballot_sync(0xffffffffu, keep && few)) >= kRaysFrom)
                    keep = keep && cull_keep_rays(v, sm.ray[warp]);
                // (the checked build walks the dropped entries too, marked, to see that no ray hits one)
                const bool walk = GEER_CHECKED ? g + lane < cnt : keep;
                const uint32_t b = __ballot_sync(0xffffffffu, walk);
                if (walk) list[n + __popc(b & lanemask_lt())] = (uint16_t)((g + lane) * 64 + (keep ? 0 : 1));
                n += __popc(b);
            }
            if (lane < kFwdUnroll) list[n + lane] = (uint16_t)(kBatch * 64);
            __syncwarp();
            walk_entries<SPLAT>(sm.rec, list, n, n_list, misc, hit_b, p, log2_amin, dx, dy, dz, f);
        }
        // a checkpoint for the backward: every ray's (T, C) in front of tile-list
        // entry n_list + cnt and where that entry's search starts in the super-tile list
        // (its state lives in shared memory, advanced by thread 0 after the next
        // barrier: the walk's registers are at their limit)
        const uint32_t nck = sm.nck;
        const bool ck = n_list + (uint32_t)cnt >= sm.next_ck && nck < (uint32_t)kCkptMax;
        if (ck) ckpt[(size_t)nck * kTilePix + fwd_ray(tid)] = make_float4(f.T, f.cr, f.cg, f.cb);
        // the tile's last contributor so far and where it lies in the super-tile list
        const uint32_t wl = __reduce_max_sync(0xffffffffu, f.last);
        if ((tid & 31) == 0) atomicMax(&sm.maxlast, wl);
        __syncthreads();
        if (ck && tid == 0) {
            ckpt_at[nck] = make_uint2(n_list + (uint32_t)cnt, sm.pos[cnt - 1] + 1u);
            sm.ckB[nck] = n_list + (uint32_t)cnt;
            sm.pend = nck + 1u;
            sm.nck = nck + 1u;
            sm.next_ck = n_list + (uint32_t)cnt + kCkptStride;
        }
        if (tid == 0 && sm.maxlast > n_list) sm.walkpos = sm.pos[sm.maxlast - 1u - n_list] + 1u;
        // the batch's hit bytes, for the backward's skip of entries its warp never hit,
        // and its item ids: the backward reads the tile's list from here without
        // filtering; with checkpoints, the count of the backward's steps (one per
        // entry and warp that hit it), summed over the block at each checkpoint
        uint32_t we = 0;
        for (int r = tid; r < cnt; r += kThreads) {
            const uint2 h = sm.hit[r];
            if (ckpt) we += (uint32_t)(__popc(__vcmpne4(h.x, 0u)) + __popc(__vcmpne4(h.y, 0u))) >> 3;
            if (hit_rec && (int64_t)n_list + r < hit_entries) {
                hit_rec[n_list + r] = h;
                id_rec[n_list + r] = sm.id[r];
            }
        }
        if (ckpt) {  // the thread's count lives in shared memory: the walk's registers are at their limit
            we += sm.wacc[tid];
            sm.wacc[tid] = we;
            if (ck) {
                we = __reduce_add_sync(0xffffffffu, we);
                if ((tid & 31) == 0) atomicAdd(&sm.work, we);
            }
        }
        shift_list(sm.id, sm.pos, cnt, s_cnt);
        // after shift_list's barrier: the checkpoint's count has landed
        if (tid == 0 && sm.pend) {
            sm.ckw[sm.pend - 1u] = sm.work;
            sm.work = 0u;
            sm.pend = 0u;
        }
        n_list += (uint32_t)cnt;
    }
    if (!f.done) f.n_eval = n_list;  // a ray that never terminated evaluated every entry walked
    if (ckpt) {
        const uint32_t we = __reduce_add_sync(0xffffffffu, sm.wacc[tid]);
        if ((tid & 31) == 0) atomicAdd(&sm.work, we);
    }
    __syncthreads();
}

// The block's rays and tile: camera, tile coordinates, ray direction (from the
// per-pixel (sin, cos) tables of the BEAP angles), the tile's association
// table entries and super-tile list. Returns false for a padding tile.
struct TileRay {
    int x, y;
    bool inside;
    float dx, dy, dz;
    TileList tl;
};

__device__ __forceinline__ bool tile_ray(const DevCam &cam, int t, const float2 *__restrict__ ptab,
                                         const uint2 *__restrict__ srange, const uint32_t *svals,
                                         const uint32_t *smask, const uint32_t *sany, int S, TileRay &r, int ray) {
    const int lt = t - cam.tile_base;
    if (lt >= cam.tiles_x * cam.tiles_y) return false;  // padding tile of a camera slot
    const int cy = lt / cam.tiles_x, cx = lt - cy * cam.tiles_x;
    r.x = cx * kTile + (ray & (kTile - 1));
    r.y = cy * kTile + ray / kTile;
    r.inside = r.x < cam.width && r.y < cam.height;
    r.dx = 0.0f;
    r.dy = 0.0f;
    r.dz = 1.0f;
    if (r.inside) {
        const float2 th = ptab[cam.pcol_off + r.x];  // (sin theta, cos theta)
        const float2 ph = ptab[cam.prow_off + r.y];  // (sin phi, cos phi)
        r.dx = th.x * ph.y;
        r.dy = th.y * ph.x;
        r.dz = th.y * ph.y;
    }
    const int sx = cx / S, sy = cy / S, bit = (cy - sy * S) * S + (cx - sx * S);
    r.tl.vals = svals;
    r.tl.words = mask_words(S);
    r.tl.mask = smask + (bit >> 5);
    r.tl.any = sany + (bit >> 5);
    r.tl.shift = bit & 31;
    r.tl.sr = srange[cam.stile_base + sy * cam.stiles_x + sx];
    return true;
}

// The L1 loss at one pixel, as geer_l1_loss_grad computes it over the n = 3 x
// pixels values (the mean absolute difference): dL/dC = sign(C - target) / n
// into dL, |C - target| added to acc.
__device__ __forceinline__ void l1_pixel(float c0, float c1, float c2, const float *__restrict__ target,
                                         float *__restrict__ dL, int64_t pix, float inv_m, float &acc) {
    const float c[3] = {c0, c1, c2};
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) {
        const float d = c[ch] - target[3 * pix + ch];
        dL[3 * pix + ch] = d > 0.0f ? inv_m : (d < 0.0f ? -inv_m : 0.0f);
        acc += fabsf(d);
    }
}

// One tile of the forward (the body of k_render_fwd): the tile's rays walk its
// list and write their colour, transmittance, last contributor and counts, the
// hit and list records, the checkpoints and the backward's unit record. With
// L1, each pixel's L1 gradient against target too (dL; |differences| summed
// into l1acc). Returns the tile's backward unit count in thread 0.
template <bool SPLAT, bool L1>
__device__ __forceinline__ uint32_t fwd_tile(WalkSmem &sm, uint32_t t_id,
                                         const DevCam *__restrict__ cams,
                                         int ncams,
                                         const float2 *__restrict__ ptab,
                                         int S,
                                         uint2 *__restrict__ tile_walk,
                                         const uint2 *__restrict__ srange,
                                         const uint32_t *__restrict__ svals,
                                         const uint32_t *__restrict__ smask,
                                         const uint32_t *__restrict__ sany,
                                         const Record *__restrict__ rec,
                                         uint32_t *__restrict__ misc,
                                         Params p,
                                         float *__restrict__ rgb,
                                         float *__restrict__ Tout,
                                         float *__restrict__ Tfin,
                                         uint32_t *__restrict__ last_out,
                                         uint2 *__restrict__ evals,
                                         uint2 *__restrict__ hit,
                                         uint32_t *__restrict__ idrec,
                                         int64_t hit_entries,
                                         const uint8_t *__restrict__ tile_mask,
                                         int64_t ntiles,
                                         uint64_t items,
                                         int64_t cap_pairs,
                                         float4 *__restrict__ ckpt,
                                         uint2 *__restrict__ ckpt_at,
                                         uint32_t *__restrict__ ckpt_cnt,
                                         uint4 *__restrict__ unit_rec,
                                         float4 *__restrict__ Cfin,
                                         const float *__restrict__ target, float *__restrict__ dL, float inv_m,
                                         float &l1acc) {
    if (!in_bounds(t_id, (uint64_t)ntiles, kSiteFwdTile, misc)) return 0u;  // block-uniform
    const int t = (int)t_id;
    if (threadIdx.x == 0) sm.cam = find_cam(cams, ncams, t);
    __syncthreads();
    const DevCam &cam = cams[sm.cam];
    TileRay tr;
    if (!tile_ray(cam, t, ptab, srange, svals, smask, sany, S, tr, fwd_ray((int)threadIdx.x))) {
        if (threadIdx.x == 0) {
            tile_walk[t] = make_uint2(0u, 0u);
            if (ckpt_cnt) ckpt_cnt[t] = 0u;
            if (unit_rec) unit_rec[t] = make_uint4(0u, 0u, 0u, 0u);
        }
        return 0u;
    }
    tr.tl.sr = checked_range(tr.tl.sr, cap_pairs, kSiteFwdList, misc);
    if (tile_mask && !tile_mask[t]) {  // another part's tile: zeros, nothing for the backward to walk
        if (threadIdx.x == 0) {
            tile_walk[t] = make_uint2(0u, 0u);
            if (ckpt_cnt) ckpt_cnt[t] = 0u;
            if (unit_rec) unit_rec[t] = make_uint4(0u, 0u, 0u, 0u);
        }
        if (tr.inside) {
            const int64_t pix = cam.pix_base + (int64_t)tr.y * cam.width + tr.x;
            rgb[3 * pix + 0] = 0.0f;
            rgb[3 * pix + 1] = 0.0f;
            rgb[3 * pix + 2] = 0.0f;
            if (Tout) Tout[pix] = 0.0f;
            Tfin[pix] = 0.0f;
            last_out[pix] = 0u;
            evals[pix] = make_uint2(0u, 0u);
            if (L1) l1_pixel(0.0f, 0.0f, 0.0f, target, dL, pix, inv_m, l1acc);
        }
        return 0u;
    }
    FwdRay f{1.0f, 0.0f, 0.0f, 0.0f, 0u, 0u, 0u, !tr.inside};
    if (SPLAT) {  // the ray's screen angles
        const float ts = atan2f(tr.dx, tr.dz), ps = atan2f(tr.dy, tr.dz);
        tr.dx = ts;
        tr.dy = ps;
    }
    forward_walk<SPLAT>(sm, tr.tl, rec, p, tr.dx, tr.dy, tr.dz,
                        hit ? hit + (int64_t)t * hit_entries : nullptr,
                                         hit ? idrec + (int64_t)t * hit_entries : nullptr, hit_entries, items,
                                         misc, ckpt ? ckpt + (size_t)t * kCkptMax * kTilePix : nullptr,
                                         ckpt ? ckpt_at + (size_t)t * kCkptMax : nullptr,
                                         f);
    if (threadIdx.x == 0) {
        tile_walk[t] = make_uint2(sm.walkpos, sm.maxlast);
        if (ckpt_cnt) ckpt_cnt[t] = sm.nck;
    }
    if (tr.inside) {
        const int64_t pix = cam.pix_base + (int64_t)tr.y * cam.width + tr.x;
        const float c0 = fmaf(f.T, cam.bg[0], f.cr), c1 = fmaf(f.T, cam.bg[1], f.cg), c2 = fmaf(f.T, cam.bg[2], f.cb);
        rgb[3 * pix + 0] = c0;
        rgb[3 * pix + 1] = c1;
        rgb[3 * pix + 2] = c2;
        if (Tout) Tout[pix] = f.T;
        Tfin[pix] = f.T;
        last_out[pix] = f.last;
        evals[pix] = make_uint2(f.n_eval, f.n_applied);
        if (Cfin && sm.nck) Cfin[pix] = make_float4(f.cr, f.cg, f.cb, f.T);  // the backward's colour behind
        if (L1) l1_pixel(c0, c1, c2, target, dL, pix, inv_m, l1acc);
    }
    // the backward's units: the checkpoints inside the walk [0, W) split it; thread k
    // writes unit k's schedule bucket (from the steps counted in it), thread
    // kUnitCountByte the number of units
    // (returns the number of units in thread 0)
    uint32_t units = 0;
    if (unit_rec && ((int)threadIdx.x <= kCkptMax || threadIdx.x == kUnitCountByte)) {
        const uint32_t W = sm.maxlast, nk = W > kCkptFirst ? min(sm.nck, (uint32_t)kCkptMax) : 0u;
        uint32_t m = 0;
        for (uint32_t j = 0; j < nk; ++j) m += sm.ckB[j] < W ? 1u : 0u;
        units = W > 0 ? m + 1u : 0u;
        const uint32_t k = threadIdx.x;
        uint8_t *rb = reinterpret_cast<uint8_t *>(unit_rec + t);
        if (k == (uint32_t)kUnitCountByte) {
            rb[k] = (uint8_t)units;
        } else if (k < units) {
            const uint32_t wlo = k == 0 ? 0u : sm.ckw[k - 1], whi = k < m ? sm.ckw[k] : sm.work;
            rb[k] = (uint8_t)order_bucket(max(whi - wlo, 1u));
        }
    }
    return units;
}

template <bool SPLAT>
__global__ void __launch_bounds__(kTilePix, GEER_FWD_MINB) k_render_fwd(const DevCam *__restrict__ cams, int ncams,
                                                            const float2 *__restrict__ ptab,
                                         int S,
                                                            uint2 *__restrict__ tile_walk,
                                                            const uint32_t *__restrict__ tile_order,
                                                            const uint2 *__restrict__ srange,
                                                            const uint32_t *__restrict__ svals,
                                                            const uint32_t *__restrict__ smask,
                                                            const uint32_t *__restrict__ sany,
                                                            const Record *__restrict__ rec,
                                                            uint32_t *__restrict__ misc, Params p,
                                                            float *__restrict__ rgb,
                                                            float *__restrict__ Tout, float *__restrict__ Tfin,
                                                            uint32_t *__restrict__ last_out,
                                                            uint2 *__restrict__ evals, uint2 *__restrict__ hit,
                                                            uint32_t *__restrict__ idrec, int64_t hit_entries,
                                                            const uint8_t *__restrict__ tile_mask, int64_t ntiles,
                                                            uint64_t items, int64_t cap_pairs,
                                                            float4 *__restrict__ ckpt, uint2 *__restrict__ ckpt_at,
                                                            uint32_t *__restrict__ ckpt_cnt,
                                                            uint4 *__restrict__ unit_rec,
                                                            float4 *__restrict__ Cfin) {
    grid_dep_sync();
    __shared__ WalkSmem sm;
    if (misc[kMiscStatus] & kStatusCapacity) return;
    float l1acc = 0.0f;
    fwd_tile<SPLAT, false>(sm, tile_order[blockIdx.x], cams, ncams, ptab, S, tile_walk, srange, svals, smask, sany, rec, misc, p, rgb, Tout, Tfin, last_out, evals, hit, idrec, hit_entries, tile_mask, ntiles, items, cap_pairs, ckpt, ckpt_at, ckpt_cnt, unit_rec, Cfin, nullptr, nullptr, 0.0f,
                                        l1acc);
}

// Every tile's full list (no early termination), filtered from its super-tile's
// list exactly as the renders do. With lists == NULL: count[t] = the list's
// length; else lists[off[t] + k] = entry k (off in the same array). For inspection.
__global__ void __launch_bounds__(kTilePix) k_expand_tiles(const DevCam *__restrict__ cams, int ncams,
                                                          const float2 *__restrict__ ptab, int S,
                                                          const uint2 *__restrict__ srange,
                                                          const uint32_t *__restrict__ svals,
                                                          const uint32_t *__restrict__ smask,
                                                          const uint32_t *__restrict__ sany,
                                                          const uint32_t *__restrict__ misc,
                                                          uint32_t *__restrict__ count_or_off,
                                                          uint32_t *__restrict__ lists, int64_t cap) {
    grid_dep_sync();
    __shared__ uint32_t s_id[2 * kTilePix];
    __shared__ FillSmem s_fill;
    __shared__ int s_cam;
    if (misc[kMiscStatus] & kStatusCapacity) return;
    const int t = blockIdx.x, tid = threadIdx.x;
    if (tid == 0) s_cam = find_cam(cams, ncams, t);
    __syncthreads();
    TileRay tr;
    if (!tile_ray(cams[s_cam], t, ptab, srange, svals, smask, sany, S, tr, tid)) {
        if (!lists && tid == 0) count_or_off[t] = 0u;
        return;
    }
    const int64_t off = lists ? (int64_t)count_or_off[t] : 0;
    uint32_t pos = tr.tl.sr.x, n_list = 0;
    bool sparse = false;
    int s_cnt = 0;
    while (true) {
        fill_list(tr.tl, pos, sparse, kTilePix, s_id, nullptr, s_cnt, s_fill);
        const int cnt = min(s_cnt, kTilePix);
        if (cnt == 0) break;
        if (lists)
            for (int r = tid; r < cnt; r += kTilePix)
                if (off + n_list + r < cap) lists[off + n_list + r] = s_id[r];
        __syncthreads();
        shift_list(s_id, nullptr, cnt, s_cnt);
        __syncthreads();
        n_list += (uint32_t)cnt;
    }
    if (!lists && tid == 0) count_or_off[t] = n_list;
}

// RenderCUDA backward (App. C): reverse traversal of each ray's contributors
// from the last one composited, transmittance recovered as T_i = T_{i+1}/(1-a_i),
// colour behind accumulated back to front. Per (camera, Gaussian) it accumulates
// dL/dsigma, dL/dc, dL/dW through d_u (outer product with the ray direction)
// and dL/do_u (the PreprocessCUDA part chains o_u = -W mu_c).
//
// The 16 values are reduced over the warp (reduce-scatter by shuffles, lanes 16, 8,
// 4, 2, 1 apart), over the tile's warps in shared memory, then added to global
// memory with one set of float4 atomics per (tile, Gaussian). (Added to global
// memory per warp, 2% faster, they lose precision: a Gaussian over many tiles takes
// eight times the roundings at its full sum, 5e-6 against 1e-6 of the quaternions'
// norm from run to run.) A warp walks the list entries below the last contributor
// of its rays that one of its rays hit in the forward (the forward's hit record;
// the same FP32 evaluation decides both).
// gS: the colour behind the current entry (what lies after it in the list, the
// background included) projected on dL/dC. dL/dalpha needs only this dot product,
// so the ray carries one scalar instead of the three channels.
struct BwdRay {
    float dx, dy, dz, g0, g1, g2, T, gS;
    uint32_t last;
};

// What one ray adds to the 16 accumulators of the Gaussian in (a, b, c, e), as
// factors, and the step of the ray's reverse compositing state. `act`: the ray
// walks the entry. Branch-free: a ray that does not hit selects zeros.
//   colour wgt (g0, g1, g2); sigma sig; exact dL/dW r d^T, dL/do_u o;
//   splat  o0, o1 = dL/d(theta_c, phi_c), r0, r1, r2 = dL/d(A, B, C):
//          dq/dtheta_c = -2 (A D0 + B D1), dq/dphi_c = -2 (B D0 + C D1),
//          dq/dA = D0^2, dq/dB = 2 D0 D1, dq/dC = D1^2.
struct RayGrad {
    float wgt, sig, r0, r1, r2, o0, o1, o2;
    bool act;  // whether the ray hits (wgt is 0 if it does not)
};

template <bool SPLAT>
__device__ __forceinline__ RayGrad ray_gradient(BwdRay &r, const float4 &a, const float4 &b, const float4 &c,
                                                const float4 &e, float log2_amin, float alpha_max, bool act) {
    const Eval v = SPLAT ? evaluate_splat(a, b, e, r.dx, r.dy, log2_amin)
                         : evaluate(a, b, c, e, r.dx, r.dy, r.dz, log2_amin);
    act = act && v.hit;
    const float ae = ex2(v.arg);
    const float alpha = fminf(ae, alpha_max);
    const float inv_om = rcp(1.0f - alpha);
    const float Ti = r.T * inv_om;  // transmittance in front of this Gaussian
    RayGrad g;
    const float wgt = Ti * alpha;
    g.wgt = act ? wgt : 0.0f;
    g.act = act;
    // dL/dalpha = sum_ch g_ch (T_i c_ch - S_ch / (1 - alpha)) = T_i (g . c) - (g . S) / (1 - alpha)
    const float gc = fmaf(r.g0, e.y, fmaf(r.g1, e.z, r.g2 * e.w));
    const float dLda = fmaf(Ti, gc, -r.gS * inv_om);
    if (act) {
        r.gS = fmaf(wgt, gc, r.gS);
        r.T = Ti;
    }
    const bool pass = act && ae < alpha_max;
    g.sig = pass ? dLda * ex2(v.kappa * kNegHalfLog2e) : 0.0f;  // dL/dsigma = dL/da e^{-kappa/2}
    const float dLdk = -0.5f * dLda * ae;
    if (SPLAT) {
        const float d0 = v.du0, d1 = v.du1;
        g.o0 = pass ? -2.0f * dLdk * fmaf(a.z, d0, a.w * d1) : 0.0f;
        g.o1 = pass ? -2.0f * dLdk * fmaf(a.w, d0, b.x * d1) : 0.0f;
        g.o2 = 0.0f;
        g.r0 = pass ? dLdk * (d0 * d0) : 0.0f;
        g.r1 = pass ? 2.0f * dLdk * (d0 * d1) : 0.0f;
        g.r2 = pass ? dLdk * (d1 * d1) : 0.0f;
        return g;
    }
    // with g_m = 2 m_u / |d_u|^2 (dkappa/dm_u), scaled by dL/dkappa:
    //   dL/dd_u = dL/dkappa (-(2 kappa / |d_u|^2) d_u + g_m x o_u),  dL/do_u = dL/dkappa (d_u x g_m)
    const float h = 2.0f * dLdk * v.inv_dd;
    const float gm0 = h * v.m0, gm1 = h * v.m1, gm2 = h * v.m2;
    const float sk = -h * v.kappa;
    const float r0 = sk * v.du0 + (gm1 * c.w - gm2 * c.z);
    const float r1 = sk * v.du1 + (gm2 * c.y - gm0 * c.w);
    const float r2 = sk * v.du2 + (gm0 * c.z - gm1 * c.y);
    g.r0 = pass ? r0 : 0.0f;
    g.r1 = pass ? r1 : 0.0f;
    g.r2 = pass ? r2 : 0.0f;
    g.o0 = pass ? v.du1 * gm2 - v.du2 * gm1 : 0.0f;
    g.o1 = pass ? v.du2 * gm0 - v.du0 * gm2 : 0.0f;
    g.o2 = pass ? v.du0 * gm1 - v.du1 * gm0 : 0.0f;
    return g;
}

// Warp sums of the 16 accumulator values: lane l and l ^ 1 end with the sum of one
// value, at the lane's offset in GradAcc (LanePerm::off).
//
// The exact integral's values are four rows of four: (r_k dx, r_k dy, r_k dz, o_k)
// and (wgt g0, wgt g1, wgt g2, sig). Bits 4 and 3 of the lane permute the columns,
// lane class c holding column i ^ c at place i: the lane keeps its ray's direction
// and dL/dC in that order, with a zero in column 3 and the column 3 value added
// through b (1 there, 0 elsewhere). So the first two exchanges (lanes 16 and 8
// apart) send the places the lane does not keep and add what arrives, without
// selecting what to send; only the next two (4 and 2 apart) select. That and
// packed arithmetic take ~50 instructions for the products and the sums, where
// selecting in every exchange took ~75. The tree of each value's sum is the plain
// butterfly's. (With the branch-free gradient and the warps' entry lists: the
// 1M-Gaussian training step 1010 -> 927 us, the surround step 21.0 -> 19.35 ms.)
//
// A product with zero does not mask an infinity or NaN, which would reach the sums of
// another column and those of entries that the ray does not hit. ODD selects instead:
// for the warps where a ray's dL/dC or colour behind is not finite, or large enough for
// a product to overflow, and from a batch with a Gaussian of such a colour on.
// (Selecting always: 1029 us for the 1M-Gaussian training step, where both sets of sums
// beside each other take 844, as one did.)
struct LanePerm {
    float2 d01, d23, b01, b23, g01, g23;
    int off;
};

template <bool SPLAT>
__device__ __forceinline__ LanePerm lane_perm(const BwdRay &r) {
    const int lane = threadIdx.x & 31, c = SPLAT ? 0 : lane >> 3;
    const auto pick = [&](int i, float a0, float a1, float a2, float a3) {
        const int k = i ^ c;
        return k == 0 ? a0 : k == 1 ? a1 : k == 2 ? a2 : a3;
    };
    LanePerm q;
    q.d01 = make_float2(pick(0, r.dx, r.dy, r.dz, 0.0f), pick(1, r.dx, r.dy, r.dz, 0.0f));
    q.d23 = make_float2(pick(2, r.dx, r.dy, r.dz, 0.0f), pick(3, r.dx, r.dy, r.dz, 0.0f));
    q.g01 = make_float2(pick(0, r.g0, r.g1, r.g2, 0.0f), pick(1, r.g0, r.g1, r.g2, 0.0f));
    q.g23 = make_float2(pick(2, r.g0, r.g1, r.g2, 0.0f), pick(3, r.g0, r.g1, r.g2, 0.0f));
    q.b01 = make_float2(pick(0, 0.0f, 0.0f, 0.0f, 1.0f), pick(1, 0.0f, 0.0f, 0.0f, 1.0f));
    q.b23 = make_float2(pick(2, 0.0f, 0.0f, 0.0f, 1.0f), pick(3, 0.0f, 0.0f, 0.0f, 1.0f));
    const int row = (lane >> 1) & 3;
    q.off = SPLAT ? lane >> 1 : row < 3 ? (c < 3 ? 4 + 3 * row + c : 13 + row) : (c < 3 ? 1 + c : 0);
    return q;
}

__device__ __forceinline__ float2 xchg2(float2 keep, float2 send, int w) {
    return add2(keep, make_float2(__shfl_xor_sync(0xffffffffu, send.x, w), __shfl_xor_sync(0xffffffffu, send.y, w)));
}

template <bool SPLAT, bool ODD>
__device__ __forceinline__ float warp_sum(const RayGrad &g, const BwdRay &r, const LanePerm &q) {
    const int lane = threadIdx.x & 31;
    if (SPLAT) {
        float v[16];
        v[0] = g.sig;
        v[1] = ODD && !g.act ? 0.0f : g.wgt * r.g0;
        v[2] = ODD && !g.act ? 0.0f : g.wgt * r.g1;
        v[3] = ODD && !g.act ? 0.0f : g.wgt * r.g2;
        v[4] = g.o0; v[5] = g.o1; v[6] = g.r0; v[7] = g.r1; v[8] = g.r2;
#pragma unroll
        for (int k = 9; k < 16; ++k) v[k] = 0.0f;
#pragma unroll
        for (int w = 8; w > 0; w >>= 1) {  // lanes with bit 2w keep the upper w values
            const bool up = lane & (2 * w);
#pragma unroll
            for (int k = 0; k < w; ++k) {
                const float send = up ? v[k] : v[k + w];
                const float keep = up ? v[k + w] : v[k];
                v[k] = keep + __shfl_xor_sync(0xffffffffu, send, 2 * w);
            }
        }
        return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
    }
    const float row[4] = {g.r0, g.r1, g.r2, g.wgt}, last[4] = {g.o0, g.o1, g.o2, g.sig};
    float2 x[2];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float2 f = make_float2(row[k], row[k]), l = make_float2(last[k], last[k]);
        float2 a, b;
        if (!ODD) {
            a = fma2(f, k < 3 ? q.d01 : q.g01, mul2(l, q.b01));
            b = fma2(f, k < 3 ? q.d23 : q.g23, mul2(l, q.b23));
        } else {
            a = mul2(f, k < 3 ? q.d01 : q.g01);
            b = mul2(f, k < 3 ? q.d23 : q.g23);
            if (k == 3 && !g.act) a = b = make_float2(0.0f, 0.0f);
            a.x = q.b01.x != 0.0f ? l.x : a.x;
            a.y = q.b01.y != 0.0f ? l.x : a.y;
            b.x = q.b23.x != 0.0f ? l.x : b.x;
            b.y = q.b23.y != 0.0f ? l.x : b.y;
        }
        const float2 v = xchg2(a, b, 16);
        const float s = v.x + __shfl_xor_sync(0xffffffffu, v.y, 8);
        if (k & 1) x[k >> 1].y = s;
        else x[k >> 1].x = s;
    }
    const bool u4 = lane & 4, u2 = lane & 2;
    const float2 y = xchg2(u4 ? x[1] : x[0], u4 ? x[0] : x[1], 4);
    const float z = (u2 ? y.y : y.x) + __shfl_xor_sync(0xffffffffu, u2 ? y.x : y.y, 2);
    return z + __shfl_xor_sync(0xffffffffu, z, 1);
}

// A backward unit's walk: tile-list entries [lo, walk.y) read back to front,
// filtered as in the forward from super-list positions [plo, walk.x) (walk.x:
// just past entry walk.y - 1; plo: where entry lo's search starts).
template <bool SPLAT, bool CG>
__device__ __forceinline__ void backward_walk(WalkSmem &sm, const TileList &tl, const Record *__restrict__ rec,
                                              const Params &p, uint32_t plo, uint32_t lo, uint2 walk,
                                              uint32_t warp_last, uint32_t block_last,
                                              const uint2 *__restrict__ hit_rec,
                                              const uint32_t *__restrict__ id_rec, int64_t hit_entries,
                                              BwdRay &ray, GradAcc *__restrict__ gacc, uint64_t items,
                                              uint32_t *misc) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float log2_amin = log2f(p.alpha_min);
    const LanePerm perm = lane_perm<SPLAT>(ray);
    const auto odd_value = [](float x) { return !(fabsf(x) < 1e15f); };
    // entry r of a batch has list index top - 1 - r
    uint32_t pos = walk.x, top = walk.y;
    int s_cnt = 0;
    while (top > lo) {
        // within the forward's record the list is read directly, beyond it filtered again
        const bool direct = id_rec && (int64_t)top <= hit_entries;
        int cnt;
        if (direct) {
            cnt = (int)min((uint32_t)kBatch, top - lo);
        } else {
            fill_list_rev(tl, pos, plo, sm.id, s_cnt, sm.fill.wcnt[0]);
            cnt = min(s_cnt, kBatch);
            if (cnt == 0) break;
        }
        // entries at or beyond the block's last contributor are not walked
        const int skip = top > block_last ? (int)min((uint32_t)cnt, top - block_last) : 0;
        if (tid >= skip && tid < cnt) {
            const uint32_t j = top - 1u - (uint32_t)tid;
            uint32_t id;
            if (direct) {
                id = ld_cg<CG>(id_rec + j);
                sm.id[tid] = id;
            } else {
                id = sm.id[tid];
            }
            // beyond the recorded entries every warp evaluates
            uint2 h = hit_rec && (int64_t)j < hit_entries ? ld_cg<CG>(hit_rec + j) : make_uint2(~0u, ~0u);
            if ((h.x | h.y) && !in_bounds(id, items, kSiteBwdItem, misc)) h = make_uint2(0u, 0u);
            // an entry no warp hit is never read: its record is not staged
            if (h.x | h.y) {
                const float4 *src = reinterpret_cast<const float4 *>(rec + id);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float4 v = src[k];
                    sm.rec[tid * 4 + k] = v;
                    if (!SPLAT && k == 3 && odd_value(v.y + v.z + v.w)) sm.odd = 1u;
                }
            }
            sm.hit[tid] = h;
        }
        for (int i = skip * 17 + tid; i < cnt * 17; i += kTilePix) (&sm.acc[0][0])[i] = 0.0f;
        __syncthreads();
        // this warp's entries: those its rays hit in the forward, below their last
        // contributor (the same FP32 decisions here would not hit the others either)
        uint8_t *const list = sm.blist[warp];
        const int first = max(skip, top > warp_last ? (int)min((uint32_t)cnt, top - warp_last) : 0);
        const int reach = top > ray.last ? (int)min((uint32_t)kBatch, top - ray.last) : 0;  // the ray's first entry
        int n = 0;
        if (direct) {
            for (int base = first & ~31; base < cnt; base += 32) {
                const int r = base + lane;
                const bool mine = r >= first && r < cnt && reinterpret_cast<const uint8_t *>(sm.hit + r)[warp] != 0;
                const uint32_t b = __ballot_sync(0xffffffffu, mine);
                if (mine) list[n + __popc(b & lanemask_lt())] = (uint8_t)r;
                n += __popc(b);
            }
        } else {
            // beyond the record: the entries that one of the warp's rays hits, four
            // evaluated together (the gradient of an entry that none hits costs three
            // times its evaluation: 764K specks on 30 tiles 33 ms with it, 17 before the
            // warps had lists, 9.6 now)
            constexpr int U = 4;
            for (int r0 = first; r0 < cnt; r0 += U) {
                bool any[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int r = min(r0 + u, cnt - 1);
                    const float4 a = sm.rec[r * 4 + 0], b = sm.rec[r * 4 + 1], c = sm.rec[r * 4 + 2], e = sm.rec[r * 4 + 3];
                    const Eval v = SPLAT ? evaluate_splat(a, b, e, ray.dx, ray.dy, log2_amin)
                                         : evaluate(a, b, c, e, ray.dx, ray.dy, ray.dz, log2_amin);
                    any[u] = v.hit && r >= reach && r0 + u < cnt && reinterpret_cast<const uint8_t *>(sm.hit + r)[warp] != 0;
                }
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (__any_sync(0xffffffffu, any[u])) {
                        if (lane == 0) list[n] = (uint8_t)(r0 + u);
                        ++n;
                    }
            }
        }
        __syncwarp();
        const auto walk_list = [&](auto odd_sums) {
            for (int k = 0; k < n; ++k) {
                const int r = (int)list[k];
                const float4 a = sm.rec[r * 4 + 0];
                const float4 b = sm.rec[r * 4 + 1];
                const float4 c = sm.rec[r * 4 + 2];
                const float4 e = sm.rec[r * 4 + 3];
                const RayGrad g = ray_gradient<SPLAT>(ray, a, b, c, e, log2_amin, p.alpha_max, r >= reach);
                const float v = warp_sum<SPLAT, decltype(odd_sums)::value>(g, ray, perm);
                if (!(lane & 1)) atomicAdd(&sm.acc[r][perm.off], v);
            }
        };
        const bool odd = odd_value(ray.g0) || odd_value(ray.g1) || odd_value(ray.g2) || odd_value(ray.gS);
        if (__any_sync(0xffffffffu, odd) || sm.odd) walk_list(std::true_type{});
        else walk_list(std::false_type{});
        __syncthreads();
        // flush: one Gaussian of the batch per thread, four float4 atomics
        if (tid >= skip && tid < cnt && (sm.hit[tid].x | sm.hit[tid].y)) {
            const float *v = sm.acc[tid];
            float4 *dst = reinterpret_cast<float4 *>(gacc + sm.id[tid]);
            atomicAdd(dst + 0, make_float4(v[0], v[1], v[2], v[3]));
            atomicAdd(dst + 1, make_float4(v[4], v[5], v[6], v[7]));
            atomicAdd(dst + 2, make_float4(v[8], v[9], v[10], v[11]));
            atomicAdd(dst + 3, make_float4(v[12], v[13], v[14], v[15]));
        }
        if (!direct) shift_list(sm.id, nullptr, cnt, s_cnt);
        __syncthreads();  // the batch's sums and ids have been read
        top -= (uint32_t)cnt;
    }
}

// Backward ray state at the end of the forward: direction, dL/dC, final
// transmittance and last contributor; the colour behind starts with the background.
__device__ __forceinline__ BwdRay bwd_ray(const TileRay &tr, const DevCam &cam, float g0, float g1, float g2, float T,
                                          uint32_t last) {
    BwdRay r;
    r.dx = tr.dx;
    r.dy = tr.dy;
    r.dz = tr.dz;
    r.g0 = g0;
    r.g1 = g1;
    r.g2 = g2;
    r.T = T;
    r.last = last;
    r.gS = T * fmaf(g0, cam.bg[0], fmaf(g1, cam.bg[1], g2 * cam.bg[2]));
    return r;
}

// The backward in units: a tile's walk [0, W) is split at the forward's
// checkpoints B_1 < B_2 < ... below W into the units [0, B_1), [B_1, B_2), ...,
// [B_m, W), each walked back to front by one block. A unit below the top starts
// every ray that walks past it from the checkpoint's state (T in front of
// B_{k+1}, and the colour behind it, C_final - C_checkpoint + T_final bg);
// the top unit starts from the final state. The units are independent, so a
// tile's long walk runs on several SMs at once and its transmittance is
// recovered by division over one unit at most. Persistent blocks take units
// in the order of k_bwd_order (descending length) from a counter.
// One backward unit (the body of k_render_bwd's loop): unit code = tile << 4 | k. CG: read what the forward wrote through
// L2 (the fused kernel reads it in the launch that wrote it).
template <bool SPLAT, bool CG>
__device__ __forceinline__ void bwd_unit(WalkSmem &sm, uint32_t code,
                                         const DevCam *__restrict__ cams,
                                         int ncams,
                                         const float2 *__restrict__ ptab,
                                         int S,
                                         const uint2 *__restrict__ tile_walk,
                                         const uint2 *__restrict__ srange,
                                         const uint32_t *__restrict__ svals,
                                         const uint32_t *__restrict__ smask,
                                         const uint32_t *__restrict__ sany,
                                         const Record *__restrict__ rec,
                                         uint32_t *__restrict__ misc,
                                         Params p,
                                         const float *__restrict__ dL_drgb,
                                         const float *__restrict__ Tfin,
                                         const uint32_t *__restrict__ last_in,
                                         const uint2 *__restrict__ hit,
                                         const uint32_t *__restrict__ idrec,
                                         int64_t hit_entries,
                                         GradAcc *__restrict__ gacc,
                                         int64_t ntiles,
                                         uint64_t items,
                                         int64_t cap_pairs,
                                         const float4 *__restrict__ ckpt,
                                         const uint2 *__restrict__ ckpt_at,
                                         const uint32_t *__restrict__ ckpt_cnt,
                                         const float4 *__restrict__ Cfin) {
    const int tray = (int)threadIdx.x;  // the ray's index in the tile
    const uint32_t t_id = code >> 4, k = code & 15u;
    if (!in_bounds(t_id, (uint64_t)ntiles, kSiteBwdTile, misc)) return;  // block-uniform
    const int t = (int)t_id;
    if (threadIdx.x == 0) {
        sm.cam = find_cam(cams, ncams, t);
        sm.odd = 0u;
    }
    __syncthreads();
    const DevCam &cam = cams[sm.cam];
    TileRay tr;
    if (!tile_ray(cam, t, ptab, srange, svals, smask, sany, S, tr, tray)) return;
    tr.tl.sr = checked_range(tr.tl.sr, cap_pairs, kSiteBwdList, misc);
    uint2 walk = ld_cg<CG>(tile_walk + t);
    if (!in_bounds(walk.x, (uint64_t)tr.tl.sr.y + 1u, kSiteBwdList, misc)) walk = make_uint2(0u, 0u);
    // the unit: tile-list entries [lo, hi), super-list positions [plo, phi)
    uint32_t lo = 0u, plo = tr.tl.sr.x, hi = walk.y, phi = walk.x;
    bool top = true;
    const uint32_t nck = ckpt_cnt ? min(ld_cg<CG>(ckpt_cnt + t), (uint32_t)kCkptMax) : 0u;
    if (k > 0 && k <= nck) {
        const uint2 a = ld_cg<CG>(ckpt_at + (size_t)t * kCkptMax + k - 1);
        lo = a.x;
        plo = a.y;
    }
    if (k < nck) {
        const uint2 b = ld_cg<CG>(ckpt_at + (size_t)t * kCkptMax + k);
        if (b.x < walk.y) {
            hi = b.x;
            phi = b.y;
            top = false;
        }
    }
    if (!in_bounds(phi, (uint64_t)walk.x + 1u, kSiteBwdList, misc) ||
        !in_bounds(plo, (uint64_t)phi + 1u, kSiteBwdList, misc) || lo >= hi)
        return;
    float g0 = 0.0f, g1 = 0.0f, g2 = 0.0f, T = 1.0f;
    uint32_t last = 0;
    int64_t pix = 0;
    if (tr.inside) {
        pix = cam.pix_base + (int64_t)tr.y * cam.width + tr.x;
        g0 = ld_cg<CG>(dL_drgb + 3 * pix + 0);
        g1 = ld_cg<CG>(dL_drgb + 3 * pix + 1);
        g2 = ld_cg<CG>(dL_drgb + 3 * pix + 2);
        T = ld_cg<CG>(Tfin + pix);
        last = ld_cg<CG>(last_in + pix);
    }
    if (SPLAT) {  // the ray's screen angles
        const float ts = atan2f(tr.dx, tr.dz), ps = atan2f(tr.dy, tr.dz);
        tr.dx = ts;
        tr.dy = ps;
    }
    BwdRay ray = bwd_ray(tr, cam, g0, g1, g2, T, last);
    if (!top && last > hi) {
        // the ray walks past this unit: its state in front of entry hi is the forward's checkpoint
        const float4 c = ld_cg<CG>(ckpt + ((size_t)t * kCkptMax + k) * kTilePix + tray);
        const float4 cf = ld_cg<CG>(Cfin + pix);
        ray.T = c.x;
        const float S0 = fmaf(T, cam.bg[0], cf.x - c.y), S1 = fmaf(T, cam.bg[1], cf.y - c.z),
                    S2 = fmaf(T, cam.bg[2], cf.z - c.w);
        ray.gS = fmaf(g0, S0, fmaf(g1, S1, g2 * S2));
    }
    const uint32_t warp_last = __reduce_max_sync(0xffffffffu, last);
    if ((threadIdx.x & 31) == 0) atomicMax(&sm.maxlast, warp_last);
    __syncthreads();
    const uint32_t block_last = sm.maxlast;
    if (block_last <= lo) return;
    backward_walk<SPLAT, CG>(sm, tr.tl, rec, p, plo, lo, make_uint2(phi, hi), warp_last, block_last,
                             hit ? hit + (int64_t)t * hit_entries : nullptr,
                             hit ? idrec + (int64_t)t * hit_entries : nullptr, hit_entries, ray, gacc, items, misc);
}

template <bool SPLAT>
__global__ void __launch_bounds__(kTilePix, GEER_BWD_MINB) k_render_bwd(const DevCam *__restrict__ cams, int ncams,
                                                                           const float2 *__restrict__ ptab,
                                         int S,
                                                                           const uint2 *__restrict__ tile_walk,
                                                                           const uint32_t *__restrict__ units,
                                                                           const uint2 *__restrict__ srange,
                                                                           const uint32_t *__restrict__ svals,
                                                                           const uint32_t *__restrict__ smask,
                                                                           const uint32_t *__restrict__ sany,
                                                                           const Record *__restrict__ rec,
                                                                           uint32_t *__restrict__ misc, Params p,
                                                                           const float *__restrict__ dL_drgb,
                                                                           const float *__restrict__ Tfin,
                                                                           const uint32_t *__restrict__ last_in,
                                                                           const uint2 *__restrict__ hit,
                                                                           const uint32_t *__restrict__ idrec,
                                                                           int64_t hit_entries,
                                                                           GradAcc *__restrict__ gacc, int64_t ntiles,
                                                                           uint64_t items, int64_t cap_pairs,
                                                                           const float4 *__restrict__ ckpt,
                                                                           const uint2 *__restrict__ ckpt_at,
                                                                           const uint32_t *__restrict__ ckpt_cnt,
                                                                           const float4 *__restrict__ Cfin) {
    grid_dep_sync();
    __shared__ WalkSmem sm;
    __shared__ uint32_t s_unit;
    if (misc[kMiscStatus] & kStatusCapacity) return;
    const uint32_t n_work = misc[kMiscUnits];
    while (true) {
        __syncthreads();  // the previous unit's shared state has been read
        if (threadIdx.x == 0) {
            s_unit = atomicAdd(&misc[kMiscUnitNext], 1u);
            sm.maxlast = 0u;
        }
        __syncthreads();
        const uint32_t w = s_unit;
        if (w >= n_work) break;
        bwd_unit<SPLAT, false>(sm, units[w], cams, ncams, ptab, S, tile_walk, srange, svals, smask, sany, rec, misc, p, dL_drgb, Tfin, last_in, hit, idrec, hit_entries, gacc, ntiles, items, cap_pairs, ckpt, ckpt_at, ckpt_cnt, Cfin);
    }
}

// Forward, L1 gradient and the render stage of the backward in one persistent
// launch (a training step's render with the per-pixel L1 loss: a tile's
// gradient needs only its own pixels, so its backward can start when its
// forward ends). Blocks take forward tiles in the render order; a finished tile
// publishes its backward units (tile << 4 | k) in a queue. Once every tile is
// taken, blocks take queue slots in order and wait, bounded, for the units of
// tiles still rendering: the backward of the finished tiles fills the SMs the
// heaviest tiles' walks leave idle. A block waits only for work that a running
// block holds. A unit's tile data, written in this launch, is read through L2
// after the slot's acquire.
constexpr uint32_t kQueueEmpty = 0xffffffffu;  // an unpublished queue slot (the host fills the queue with it)
constexpr uint32_t kQueuePolls = 1u << 22;     // bound of a wait for a queue slot (<= ~1 us sleep between polls)

template <bool SPLAT>
__global__ void __launch_bounds__(kTilePix, GEER_BWD_MINB) k_render_train(
    const DevCam *__restrict__ cams, int ncams, const float2 *__restrict__ ptab,
                                         int S, uint2 *__restrict__ tile_walk, const uint32_t *__restrict__ tile_order, const uint2 *__restrict__ srange,
    const uint32_t *__restrict__ svals, const uint32_t *__restrict__ smask, const uint32_t *__restrict__ sany,
    const Record *__restrict__ rec,
    uint32_t *__restrict__ misc, Params p, float *__restrict__ rgb, float *__restrict__ Tout,
    float *__restrict__ Tfin, uint32_t *__restrict__ last, uint2 *__restrict__ evals, uint2 *__restrict__ hit,
    uint32_t *__restrict__ idrec, int64_t hit_entries, const uint8_t *__restrict__ tile_mask, int64_t ntiles,
    uint64_t items, int64_t cap_pairs, float4 *__restrict__ ckpt, uint2 *__restrict__ ckpt_at,
    uint32_t *__restrict__ ckpt_cnt, uint4 *__restrict__ unit_rec, float4 *__restrict__ Cfin,
    const float *__restrict__ target, float *__restrict__ dL, float inv_m, float *__restrict__ loss,
    GradAcc *__restrict__ gacc, uint32_t *__restrict__ queue, uint32_t queue_cap) {
    grid_dep_sync();
    __shared__ WalkSmem sm;
    __shared__ uint32_t s_work;
    __shared__ float s_loss;
    if (misc[kMiscStatus] & kStatusCapacity) return;
    float l1acc = 0.0f;
    if (threadIdx.x == 0) s_loss = 0.0f;
    while (true) {  // forward tiles
        __syncthreads();  // the previous tile's shared state has been read
        if (threadIdx.x == 0) s_work = atomicAdd(&misc[kMiscFwdNext], 1u);
        __syncthreads();
        const uint32_t f = s_work;
        if (f >= (uint32_t)ntiles) break;
        const uint32_t t = tile_order[f];
        const uint32_t nu = fwd_tile<SPLAT, true>(
            sm, t, cams, ncams, ptab, S, tile_walk, srange, svals, smask, sany, rec, misc, p, rgb, Tout, Tfin, last,
            evals, hit, idrec, hit_entries, tile_mask, ntiles, items, cap_pairs, ckpt, ckpt_at, ckpt_cnt, unit_rec,
            Cfin, target, dL, inv_m, l1acc);
        __syncthreads();  // every thread's outputs of the tile are written
        if (threadIdx.x == 0) {
            __threadfence();  // release: the tile's outputs before its units
            if (nu) {
                const uint32_t slot = atomicAdd(&misc[kMiscUnitsPub], nu);
                for (uint32_t k = 0; k < nu; ++k)
                    if (slot + k < queue_cap) atomicExch(&queue[slot + k], (t << 4) | k);
            }
            __threadfence();
            atomicAdd(&misc[kMiscFwdDone], 1u);
        }
    }
    // the L1 loss: one atomic per block
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) l1acc += __shfl_xor_sync(0xffffffffu, l1acc, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(&s_loss, l1acc);
    __syncthreads();
    if (threadIdx.x == 0 && loss) atomicAdd(loss, s_loss * inv_m);
    while (true) {  // backward units, in the order they were published
        __syncthreads();  // the previous unit's shared state has been read
        if (threadIdx.x == 0) {
            const uint32_t w = atomicAdd(&misc[kMiscTrainNext], 1u);
            uint32_t code = kQueueEmpty, sleep = 32;
            for (uint32_t it = 0; w < queue_cap; ++it) {
                const uint32_t c = atomicAdd(&queue[w], 0u);
                if (c != kQueueEmpty) {
                    code = c;
                    break;
                }
                // every tile finished and published: slot w beyond the published units stays empty
                if (atomicAdd(&misc[kMiscFwdDone], 0u) >= (uint32_t)ntiles) {
                    __threadfence();  // the final unit count after the last tile's count
                    if (w >= atomicAdd(&misc[kMiscUnitsPub], 0u)) break;
                }
                if (it + 1 == kQueuePolls) {
                    atomicOr(&misc[kMiscStatus], kStatusTimeout);
                    break;
                }
                __nanosleep(sleep);
                sleep = min(sleep * 2u, 1024u);
            }
            __threadfence();  // acquire: the unit's tile data after its slot
            sm.maxlast = 0u;
            s_work = code;
        }
        __syncthreads();
        const uint32_t code = s_work;
        if (code == kQueueEmpty) break;
        bwd_unit<SPLAT, true>(sm, code, cams, ncams, ptab, S, tile_walk, srange, svals,
                                           smask, sany, rec, misc, p, dL, Tfin, last, hit, idrec, hit_entries, gacc,
                                           ntiles, items, cap_pairs, ckpt, ckpt_at, ckpt_cnt, Cfin);
    }
}

}  // namespace

cudaError_t launch_render_fwd(const geer_workspace *ws, float *rgb, float *T_final, cudaStream_t s) {
    if (ws->n_tiles == 0) return cudaSuccess;
    launch_k(ws->params.alpha_model == GEER_ALPHA_EXACT ? k_render_fwd<false> : k_render_fwd<true>,
        dim3((unsigned)ws->n_tiles), dim3(kTilePix), 0, s,
        ws->d_cams, ws->n_cams, ws->d_pix_tab, ws->super_size, ws->d_tile_walk, ws->d_tile_order,
        ws->d_srange, ws->d_vals[ws->sorted_buf], ws->d_smask[ws->sorted_buf], ws->d_sany, ws->d_rec, ws->d_misc,
        ws->params, rgb, T_final,
        ws->d_Tfin, ws->d_last, ws->d_evals, ws->d_hit, ws->d_idrec, ws->hit_entries,
        ws->tile_mask_on ? static_cast<const uint8_t *>(ws->d_tile_mask) : nullptr, ws->n_tiles,
        (uint64_t)ws->n_cams * (uint64_t)ws->n_gauss, ws->cap_pairs, ws->d_ckpt, ws->d_ckpt_at, ws->d_ckpt_cnt,
        ws->d_unit_rec, ws->d_Cfin);
    return cudaGetLastError();
}

cudaError_t launch_expand_tiles(const geer_workspace *ws, uint32_t *count_or_off, uint32_t *lists, cudaStream_t s) {
    if (ws->n_tiles == 0) return cudaSuccess;
    launch_k(k_expand_tiles, dim3((unsigned)ws->n_tiles), dim3(kTilePix), 0, s, ws->d_cams, ws->n_cams,
             ws->d_pix_tab, ws->super_size, ws->d_srange, ws->d_vals[ws->sorted_buf], ws->d_smask[ws->sorted_buf], ws->d_sany, ws->d_misc,
             count_or_off, lists, ws->cap_pairs);
    return cudaGetLastError();
}

cudaError_t launch_render_bwd(const geer_workspace *ws, const float *dL_drgb, cudaStream_t s) {
    if (ws->n_tiles == 0) return cudaSuccess;
    launch_k(ws->params.alpha_model == GEER_ALPHA_EXACT ? k_render_bwd<false> : k_render_bwd<true>,
        dim3((unsigned)std::max(1, ws->bwd_grid)), dim3(kTilePix), 0, s,
        ws->d_cams, ws->n_cams, ws->d_pix_tab, ws->super_size, ws->d_tile_walk, ws->d_bwd_order,
        ws->d_srange, ws->d_vals[ws->sorted_buf], ws->d_smask[ws->sorted_buf], ws->d_sany, ws->d_rec, ws->d_misc,
        ws->params, dL_drgb,
        ws->d_Tfin, ws->d_last, ws->d_hit, ws->d_idrec, ws->hit_entries, ws->d_gacc, ws->n_tiles,
        (uint64_t)ws->n_cams * (uint64_t)ws->n_gauss, ws->cap_pairs, ws->d_ckpt, ws->d_ckpt_at, ws->d_ckpt_cnt,
        ws->d_Cfin);
    return cudaGetLastError();
}

cudaError_t launch_render_train(const geer_workspace *ws, const float *target, float *rgb, float *T_final,
                                float *dL_drgb, float *loss, cudaStream_t s) {
    if (ws->n_tiles == 0) return cudaSuccess;
    const int64_t m = 3 * ws->n_pixels;  // the L1 mean's value count
    launch_k(ws->params.alpha_model == GEER_ALPHA_EXACT ? k_render_train<false> : k_render_train<true>,
        dim3((unsigned)std::max(1, ws->train_grid)), dim3(kTilePix), 0, s,
        ws->d_cams, ws->n_cams, ws->d_pix_tab, ws->super_size, ws->d_tile_walk, ws->d_tile_order,
        ws->d_srange, ws->d_vals[ws->sorted_buf], ws->d_smask[ws->sorted_buf], ws->d_sany, ws->d_rec, ws->d_misc, ws->params, rgb, T_final,
        ws->d_Tfin, ws->d_last, ws->d_evals, ws->d_hit, ws->d_idrec, ws->hit_entries,
        ws->tile_mask_on ? static_cast<const uint8_t *>(ws->d_tile_mask) : nullptr, ws->n_tiles,
        (uint64_t)ws->n_cams * (uint64_t)ws->n_gauss, ws->cap_pairs, ws->d_ckpt, ws->d_ckpt_at, ws->d_ckpt_cnt,
        ws->d_unit_rec, ws->d_Cfin, target, dL_drgb, m > 0 ? 1.0f / (float)m : 0.0f, loss, ws->d_gacc,
        ws->d_bwd_order, (uint32_t)(ws->n_tiles * (kCkptMax + 1)));
    return cudaGetLastError();
}

int render_train_blocks_per_sm(int alpha_model) {
    int b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &b, alpha_model == GEER_ALPHA_EXACT ? k_render_train<false> : k_render_train<true>,
            kTilePix, 0) != cudaSuccess)
        b = 1;
    return b < 1 ? 1 : b;
}

int render_bwd_blocks_per_sm(int alpha_model) {
    int b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &b, alpha_model == GEER_ALPHA_EXACT ? k_render_bwd<false> : k_render_bwd<true>, kTilePix, 0) != cudaSuccess)
        b = 1;
    return b < 1 ? 1 : b;
}

}  // namespace geer
