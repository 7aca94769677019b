// preprocess.cu -- per-Gaussian preprocessing (Algorithm 1: CullGaussian,
// ViewspaceGaussians, PBF_Intersect, PCA_Whitening), the pair-count scan and
// DuplicateWithKeys.
//
// The PBF part runs in exactly rounded FP32 operations in a fixed order
// (__fmul_rn / __fadd_rn / __fsub_rn / __fdiv_rn / __fsqrt_rn, which the
// compiler never contracts), so the tile ranges and depth keys are bit-for-bit
// reproducible by an independent FP32 implementation of the same sequence.
#include <cooperative_groups.h>

#include <algorithm>

#include "geer_internal.cuh"

namespace geer {
namespace {

__device__ __forceinline__ float fm(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fa(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float fs(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float fdv(float a, float b) { return __fdiv_rn(a, b); }
__device__ __forceinline__ float fsq(float a) { return __fsqrt_rn(a); }

// An arc of dihedral angle in half-angle-tangent space tau = tan(angle / 2)
// (the mirror transform with xi = 1, App. D.2). kind 0 empty, 1 [lo, hi],
// 2 wrapping [lo, +inf) u (-inf, hi], 3 full circle.
struct Arc {
    int kind;
    float lo, hi;
};

// tan(angle/2) of the planar direction (x, z), angle measured from +z towards +x.
__device__ float half_tan(float x, float z) {
    float r = fsq(fa(fm(x, x), fm(z, z)));
    return fdv(z >= 0.0f ? x : fs(r, z), z >= 0.0f ? fa(r, z) : x);  // x / (r + z) or (r - z) / x
}

// PBF bounds about one camera axis (Sec. 3.2, App. D.1): the bounding planes
// through the axis have tangent c solving T22 c^2 - 2 T02 c + T00 = 0 with
// T = lambda^2 Sigma_c - mu_c mu_c^T. The discriminant T02^2 - T00 T22 equals
// lambda^2 (P - lambda^2 D) with P = mu^T adj(Sigma_pp) mu and D = det(Sigma_pp),
// evaluated without cancellation. No real root: the axis pierces the ellipsoid
// and the arc is the full circle (clamp to the full FoV, App. D.1). The four
// mirrored candidates are reduced to the two nearest the centre's mirrored
// angle (App. D.2) and widened by a 2^-18 (1 + tau^2) margin.
__device__ Arc pbf_arc(float mx, float mz, float T00, float T02, float T22, float P, float D, float lam2) {
    Arc a{3, 0.0f, 0.0f};
    float disc = fm(lam2, fs(P, fm(lam2, D)));
    if (!(disc > 0.0f)) return a;
    float sq = fsq(disc);
    float qq = fa(T02, (T02 >= 0.0f) ? sq : -sq);
    if (qq == 0.0f) return a;
    float cand[4];
    cand[0] = half_tan(qq, T22);
    cand[1] = half_tan(-qq, -T22);
    cand[2] = half_tan(T00, qq);
    cand[3] = half_tan(-T00, -qq);
    float tm = half_tan(mx, mz);
    if (!isfinite(tm)) return a;
#pragma unroll
    for (int i = 0; i < 4; ++i)
        if (!isfinite(cand[i])) return a;
    bool have_lo = false, have_hi = false;
    float lo = 0.0f, hi = 0.0f, mn = cand[0], mxv = cand[0];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float v = cand[i];
        if (v < mn) mn = v;
        if (v > mxv) mxv = v;
        if (v < tm && (!have_lo || v > lo)) { lo = v; have_lo = true; }
        if (v > tm && (!have_hi || v < hi)) { hi = v; have_hi = true; }
    }
    a.kind = 1;
    if (!have_hi) { hi = mn; a.kind = 2; }
    if (!have_lo) { lo = mxv; a.kind = 2; }
    const float margin = 3.814697265625e-06f;  // 2^-18
    a.lo = fs(lo, fm(margin, fa(1.0f, fm(lo, lo))));
    a.hi = fa(hi, fm(margin, fa(1.0f, fm(hi, hi))));
    return a;
}

// The arc rotated by pi (tau -> -1/tau), for rays whose other BEAP angle is
// beyond 90 degrees.
__device__ Arc shift_arc(Arc a) {
    Arc r = a;
    if (a.kind == 0 || a.kind == 3) return r;
    if (a.lo == 0.0f || a.hi == 0.0f) { r.kind = 3; return r; }
    r.lo = fdv(-1.0f, a.lo);
    r.hi = fdv(-1.0f, a.hi);
    if (a.kind == 2) r.kind = 1;
    else r.kind = (a.lo < 0.0f && a.hi > 0.0f) ? 2 : 1;
    return r;
}

// The first tile index k in [0, n] with pred(v(k)) (false before, true from k on:
// pred is monotone in k), searched from a guess k in [0, n]; below: v(k - 1), at: v(k)
// (anything where there is none). The guess only sets where the probes start, so the
// result is exactly the first true index whatever the guess.
template <typename Value, typename Pred>
__device__ __forceinline__ int first_true_from(int k, int n, float below, float at, Value value, Pred pred) {
    if (k > 0 && pred(below)) {
        do --k;
        while (k > 0 && pred(value(k - 1)));
    } else if (k < n && !pred(at)) {
        do ++k;
        while (k < n && !pred(value(k)));
    }
    return k;
}

// atan(x) within 2e-5 rad, on [-1, 1] by Abramowitz and Stegun 4.4.49, pi/2 - atan(1/x)
// beyond. Only for where a search starts.
__device__ __forceinline__ float atan_guess(float x) {
    const float ax = fabsf(x), t = ax > 1.0f ? __fdividef(1.0f, ax) : ax, u = t * t;
    const float y = t * fmaf(u, fmaf(u, fmaf(u, fmaf(u, 0.0208351f, -0.0851330f), 0.1801410f), -0.3302995f), 0.9998660f);
    return copysignf(ax > 1.0f ? 1.5707963f - y : y, x);
}

// Tile range [lo, hi) whose half-angle span [ta, tb] (tab[i].x, tab[i].y, both
// increasing in i) meets the arc; prefix u suffix becomes the whole range. BEAP
// angles are linear in the pixel index (Sec. 3.3), so the pixel of a bound tau
// is about (2 atan(tau)) * ppr + (w - 1) / 2 (ppr: pixels per radian, half: (w - 1) / 2),
// and its tile nearly always the answer: the four edges that confirm both ends are
// loaded together, and only a miss probes further.
__device__ void arc_range(Arc a, const float4 *tab, int n, float ppr, float half, int &olo, int &ohi) {
    olo = 0;
    ohi = 0;
    if (a.kind == 0) return;
    if (a.kind == 3) { ohi = n; return; }
    const float plo = fmaf(2.0f * atan_guess(a.lo), ppr, half), phi = fmaf(2.0f * atan_guess(a.hi), ppr, half);
    // first index with tb >= a.lo (tb: the tile's last ray), then first with ta > a.hi
    const int k0 = min(max((int)ceilf((plo - (kTile - 1)) / kTile), 0), n);
    const int k1 = min(max((int)floorf(phi / kTile) + 1, 0), n);
    const float b0 = tab[max(k0 - 1, 0)].y, e0 = tab[min(k0, n - 1)].y;
    const float b1 = tab[max(k1 - 1, 0)].x, e1 = tab[min(k1, n - 1)].x;
    const int first = first_true_from(k0, n, b0, e0, [&](int k) { return tab[k].y; }, [&](float v) { return v >= a.lo; });
    const int last = first_true_from(k1, n, b1, e1, [&](int k) { return tab[k].x; }, [&](float v) { return v > a.hi; }) - 1;
    if (a.kind == 1) {
        if (first <= last) { olo = first; ohi = last + 1; }
        return;
    }
    bool suf = first < n, pre = last >= 0;
    if (suf && pre) { olo = 0; ohi = n; }
    else if (suf) { olo = first; ohi = n; }
    else if (pre) { olo = 0; ohi = last + 1; }
}

// lambda^2 >= 2 ln(sigma / alpha_min) with basic operations only, times (1 + pad):
// ln m <= 2 (z + z^3 / (3 (1 - z^2))), z = (m - 1)/(m + 1), m in [1, 2).
__device__ float lambda2(float sigma, float alpha_min, float pad) {
    float x = fdv(sigma, alpha_min);
    int e;
    float m = frexpf(x, &e);
    m = fm(m, 2.0f);
    e = e - 1;
    float z = fdv(fs(m, 1.0f), fa(m, 1.0f));
    float z2 = fm(z, z);
    float t = fdv(fm(z, z2), fm(3.0f, fs(1.0f, z2)));
    float lnm = fm(2.0f, fa(z, t));
    float lnx = fa(fm((float)e, 0.693147182464599609375f), lnm);
    return fm(fm(2.0f, lnx), fa(1.0f, pad));
}

// ---- Splatting bounds (the association ablation, Sec. 4) -------------------
// The EWA and UT alternatives to PBF bound the Gaussian's projection onto the
// BEAP screen (theta, phi) = (atan2(x, z), atan2(y, z)) by a box; the box's
// angle intervals become arcs of the same half-angle-tangent form as PBF's,
// so the tile ranges and everything after them are shared. Plain FP32
// arithmetic (no reproducibility contract: the bounds are compared with an
// FP64 definition within a tolerance).
constexpr float kPiF = 3.14159265358979f, kTwoPiF = 6.28318530717959f;
constexpr float kSplatNear = 0.2f;  // near plane of the splatting pipelines
constexpr float kSqrt3 = 1.7320508075688772f;

// tan(a / 2) for a in [-pi, pi]; the half angle is kept below pi / 2 so that the
// FP32 rounding of pi cannot turn the tangent's sign at the ends.
__device__ __forceinline__ float tan_half(float a) {
    return tanf(fminf(fmaxf(0.5f * a, -1.5707962f), 1.5707962f));
}

// The arc of the angles [lo, hi] taken modulo 2 pi.
__device__ Arc angle_arc(float lo, float hi) {
    Arc a{3, 0.0f, 0.0f};
    if (!(hi - lo < kTwoPiF) || !isfinite(lo) || !isfinite(hi)) return a;
    const float k = floorf((lo + kPiF) / kTwoPiF);  // lo into [-pi, pi)
    lo -= k * kTwoPiF;
    hi -= k * kTwoPiF;
    if (hi <= kPiF) {
        a.kind = 1;
        a.lo = tan_half(lo);
        a.hi = tan_half(hi);
    } else {  // through pi: [lo, pi] u (-pi, hi - 2 pi]
        a.kind = 2;
        a.lo = tan_half(lo);
        a.hi = tan_half(hi - kTwoPiF);
    }
    return a;
}

// The splatting box of a live item as four arcs: theta (a), theta turned by pi
// (a1: rows whose rays have cos(phi) < 0 see atan2(x, z) = theta + pi), phi (b)
// and phi turned (b1). (x, y, z): camera-frame mean; column k of M: axis k;
// s: scales. EWA: Sigma_2 = J Sigma_c J^T with the rows of J the gradients of
// the two angles, summed over the axes as s_k^2 (J M_k)(J M_k)^T. UT: the six
// off-centre sigma points mu +- sqrt(3) s_k M_k, their angles taken relative to
// the mean's (atan2 of the cross and dot products with the offset split out,
// so small Gaussians lose no digits); weights 1/6 each, the centre point 0 for
// the mean and 2 for the covariance.
// The EWA factor of Sigma_2 = sum_k f_k f_k^T: f_k = s_k J M_k, J the gradients
// of the two screen angles at the mean (x, y, z).
__device__ __forceinline__ void ewa_factor(float x, float y, float z, const float M[9], const float s[3], float fx[3],
                                           float fy[3]) {
    const float rx = 1.0f / (x * x + z * z), ry = 1.0f / (y * y + z * z);
    const float ja0 = z * rx, ja2 = -x * rx, jb1 = z * ry, jb2 = -y * ry;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        fx[k] = s[k] * (ja0 * M[k] + ja2 * M[6 + k]);
        fy[k] = s[k] * (jb1 * M[3 + k] + jb2 * M[6 + k]);
    }
}

// The EWA splat of a live item for GEER_ALPHA_SPLAT: the mean's screen angles
// and the conic Sigma_2^-1 = (A, B; B, C), out = {theta, phi, A, B, C}. The
// determinant is the sum of the squared 2 x 2 minors of the factor
// (Cauchy-Binet), free of the cancellation of c00 c11 - c01^2. False when
// Sigma_2 is singular (the item is culled).
__device__ __forceinline__ bool splat_conic(float x, float y, float z, const float M[9], const float s[3],
                                            float out[5]) {
    float fx[3], fy[3];
    ewa_factor(x, y, z, M, s, fx, fy);
    float c00 = 0.0f, c01 = 0.0f, c11 = 0.0f, det = 0.0f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        c00 += fx[k] * fx[k];
        c01 += fx[k] * fy[k];
        c11 += fy[k] * fy[k];
        const int l = (k + 1) % 3;
        const float mk = fx[k] * fy[l] - fy[k] * fx[l];
        det += mk * mk;
    }
    if (!(det > 0.0f) || !isfinite(det)) return false;
    const float inv = 1.0f / det;
    out[0] = atan2f(x, z);
    out[1] = atan2f(y, z);
    out[2] = c11 * inv;
    out[3] = -c01 * inv;
    out[4] = c00 * inv;
    return isfinite(out[2]) && isfinite(out[4]);
}

__device__ __forceinline__ void splat_arcs(int mode, int snug, float amin, float sigma, float x, float y, float z,
                                           const float M[9], const float s[3], Arc &a, Arc &a1, Arc &b, Arc &b1) {
    float tc = atan2f(x, z), pc = atan2f(y, z);
    float c00 = 0.0f, c01 = 0.0f, c11 = 0.0f;
    if (mode == GEER_ASSOC_EWA) {
        float fx[3], fy[3];
        ewa_factor(x, y, z, M, s, fx, fy);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            c00 += fx[k] * fx[k];
            c01 += fx[k] * fy[k];
            c11 += fy[k] * fy[k];
        }
    } else {
        float dt[6], dp[6], mt = 0.0f, mp = 0.0f;
        const float rxz = x * x + z * z, ryz = y * y + z * z;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float f = (h == 0 ? kSqrt3 : -kSqrt3) * s[k];
                const float ox = f * M[k], oy = f * M[3 + k], oz = f * M[6 + k];
                dt[2 * k + h] = atan2f(ox * z - oz * x, rxz + ox * x + oz * z);
                dp[2 * k + h] = atan2f(oy * z - oz * y, ryz + oy * y + oz * z);
                mt += dt[2 * k + h];
                mp += dp[2 * k + h];
            }
        }
        mt *= (1.0f / 6.0f);
        mp *= (1.0f / 6.0f);
        c00 = 2.0f * mt * mt;
        c01 = 2.0f * mt * mp;
        c11 = 2.0f * mp * mp;
        float q00 = 0.0f, q01 = 0.0f, q11 = 0.0f;
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            const float et = dt[i] - mt, ep = dp[i] - mp;
            q00 += et * et;
            q01 += et * ep;
            q11 += ep * ep;
        }
        c00 += q00 * (1.0f / 6.0f);
        c01 += q01 * (1.0f / 6.0f);
        c11 += q11 * (1.0f / 6.0f);
        tc += mt;
        pc += mp;
    }
    float et, ep;
    if (snug) {  // bounding box of the alpha_min ellipse
        const float t = 2.0f * logf(sigma / amin);
        et = sqrtf(fmaxf(t * c00, 0.0f));
        ep = sqrtf(fmaxf(t * c11, 0.0f));
    } else {  // 3 sqrt of the larger eigenvalue, both axes
        const float h = 0.5f * (c00 + c11), d = 0.5f * (c00 - c11);
        et = ep = 3.0f * sqrtf(fmaxf(h + sqrtf(d * d + c01 * c01), 0.0f));
    }
    a = angle_arc(tc - et, tc + et);
    a1 = angle_arc(tc - et + kPiF, tc + et + kPiF);
    b = angle_arc(pc - ep, pc + ep);
    b1 = angle_arc(pc - ep + kPiF, pc + ep + kPiF);
}


// Real SH of degree <= 3 in the 3DGS convention (Condon-Shortley phase, index
// l^2 + l + m), written out as polynomials of the unit direction. The constants
// are K_lm sqrt(2)^(m != 0) = sqrt((2l+1)/(4 pi) (l-|m|)!/(l+|m|)!) (* sqrt 2).
template <int DEG>
__device__ __forceinline__ void sh_colour(const float *row, float x, float y, float z, float rgb[3]) {
    constexpr int deg = DEG;
    float Y[16];
    Y[0] = 0.28209479177387814f;  // 1/(2 sqrt(pi))
    if (deg >= 1) {
        const float k1 = 0.4886025119029199f;  // sqrt(3/(4 pi))
        Y[1] = -k1 * y; Y[2] = k1 * z; Y[3] = -k1 * x;
    }
    if (deg >= 2) {
        float xx = x * x, yy = y * y, zz = z * z;
        Y[4] = 1.0925484305920792f * x * y;               // sqrt(15/pi)/2
        Y[5] = -1.0925484305920792f * y * z;
        Y[6] = 0.31539156525252005f * (2.0f * zz - xx - yy);  // sqrt(5/pi)/4
        Y[7] = -1.0925484305920792f * x * z;
        Y[8] = 0.5462742152960396f * (xx - yy);           // sqrt(15/pi)/4
        if (deg >= 3) {
            Y[9] = -0.5900435899266435f * y * (3.0f * xx - yy);        // sqrt(35/(2 pi))/4
            Y[10] = 2.890611442640554f * x * y * z;                    // sqrt(105/pi)/2
            Y[11] = -0.4570457994644658f * y * (4.0f * zz - xx - yy);  // sqrt(21/(2 pi))/4
            Y[12] = 0.3731763325901154f * z * (2.0f * zz - 3.0f * xx - 3.0f * yy);  // sqrt(7/pi)/4
            Y[13] = -0.4570457994644658f * x * (4.0f * zz - xx - yy);
            Y[14] = 1.445305721320277f * z * (xx - yy);                // sqrt(105/pi)/4
            Y[15] = -0.5900435899266435f * x * (xx - 3.0f * yy);
        }
    }
    float c[3] = {0.5f, 0.5f, 0.5f};
    sh_each<DEG>(row, [&](int i, float v) { c[i % 3] += Y[i / 3] * v; });
    rgb[0] = fmaxf(c[0], 0.0f);
    rgb[1] = fmaxf(c[1], 0.0f);
    rgb[2] = fmaxf(c[2], 0.0f);
}

// True when the association predicate reduces to the rectangle X0 x Y0: no
// flipped-angle ranges and X0, Y0 inside the tiles whose rays all have
// cos(theta) >= 0 (columns) and cos(phi) >= 0 (rows).
__device__ __forceinline__ bool is_rect(const DevCam &cam, const int rg[8]) {
    if (rg[2] < rg[3] || rg[6] < rg[7]) return false;
    if (rg[0] >= rg[1] || rg[4] >= rg[5]) return true;  // empty
    return rg[0] >= cam.c0lo && rg[1] <= cam.c0hi && rg[4] >= cam.r0lo && rg[5] <= cam.r0hi;
}


// The association predicate tile_assoc(x, y) = (z_row(y) & x in X0 | w_row(y) & x in X1)
// & (z_col(x) & y in Y0 | w_col(x) & y in Y1), with the z / w flag sets of the
// camera's rows and columns (one interval / two runs, DevCam), is a union of
// products of row and column sets. Its count over a region follows in constant
// time by inclusion-exclusion, and the set itself is the union of at most nine
// rectangles.
__device__ __forceinline__ int ilen(int lo, int hi) { return hi > lo ? hi - lo : 0; }

// Members of [lo, hi) in a flag set: kind 0 the z interval, 1 the w runs, 2 both.
__device__ __forceinline__ int flag_count(int lo, int hi, const int32_t z[2], const int32_t w[2], int kind) {
    if (kind == 0) return ilen(max(lo, z[0]), min(hi, z[1]));
    int alo = lo, ahi = min(hi, w[0]), blo = max(lo, w[1]), bhi = hi;
    if (kind == 2) {
        alo = max(alo, z[0]);
        ahi = min(ahi, z[1]);
        blo = max(blo, z[0]);
        bhi = min(bhi, z[1]);
    }
    return ilen(alo, ahi) + ilen(blo, bhi);
}

// Associated tiles of the item with ranges rg in [x0, x1) x [y0, y1).
__device__ __forceinline__ uint32_t assoc_count(const DevCam &cam, const int rg[8], int x0, int x1, int y0, int y1) {
    // column sets of the terms a0 (X0), a1 (X1), a0 a1; row sets of b0 (Y0), b1 (Y1), b0 b1
    const int alo[3] = {rg[0], rg[2], max(rg[0], rg[2])}, ahi[3] = {rg[1], rg[3], min(rg[1], rg[3])};
    const int blo[3] = {rg[4], rg[6], max(rg[4], rg[6])}, bhi[3] = {rg[5], rg[7], min(rg[5], rg[7])};
    int64_t total = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            // rows with the flag of term i inside Y_j, columns with the flag of term j inside X_i
            const int rows = flag_count(max(y0, blo[j]), min(y1, bhi[j]), cam.zr, cam.wr, i);
            if (rows == 0) continue;
            const int cols = flag_count(max(x0, alo[i]), min(x1, ahi[i]), cam.zc, cam.wc, j);
            const int sg = (i == 2) != (j == 2) ? -1 : 1;
            total += (int64_t)sg * rows * cols;
        }
    }
    return (uint32_t)total;
}

// The associated set as rectangles {x0, x1, y0, y1} (at most nine, overlapping
// only on rows / columns that carry both flags): calls f for each.
template <typename F>
__device__ __forceinline__ void assoc_rects(const DevCam &cam, const int rg[8], F f) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {      // rows of the z interval (i = 0) or the w runs (i = 1) ...
#pragma unroll
        for (int j = 0; j < 2; ++j) {  // ... crossed with columns of the z interval or the w runs
            const int xlo = rg[2 * i], xhi = rg[2 * i + 1];      // X_i
            const int ylo = rg[4 + 2 * j], yhi = rg[5 + 2 * j];  // Y_j
            if (xlo >= xhi || ylo >= yhi) continue;
#pragma unroll
            for (int ri = 0; ri < 2; ++ri) {
                if (i == 0 && ri == 1) break;
                const int r0 = i == 0 ? cam.zr[0] : (ri == 0 ? 0 : cam.wr[1]);
                const int r1 = i == 0 ? cam.zr[1] : (ri == 0 ? cam.wr[0] : cam.tiles_y);
                const int y0 = max(ylo, r0), y1 = min(yhi, r1);
                if (y0 >= y1) continue;
#pragma unroll
                for (int ci = 0; ci < 2; ++ci) {
                    if (j == 0 && ci == 1) break;
                    const int c0 = j == 0 ? cam.zc[0] : (ci == 0 ? 0 : cam.wc[1]);
                    const int c1 = j == 0 ? cam.zc[1] : (ci == 0 ? cam.wc[0] : cam.tiles_x);
                    const int x0 = max(xlo, c0), x1 = min(xhi, c1);
                    if (x0 < x1) f(make_int4(x0, x1, y0, y1));
                }
            }
        }
    }
}

// Block-wide exclusive scan (256 threads); returns the exclusive prefix and the block total.
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t x, uint32_t *wsum, uint32_t &total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t v = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
    }
    if (lane == 31) wsum[warp] = v;
    __syncthreads();
    uint32_t pre = 0, tot = 0;
#pragma unroll
    for (int w = 0; w < kPrepThreads / 32; ++w) {
        const uint32_t t = wsum[w];
        pre += w < warp ? t : 0u;
        tot += t;
    }
    __syncthreads();
    total = tot;
    return pre + v - x;
}

// Thread per Gaussian, loop over cameras (the Gaussian's parameters are read once).
// Bound by issued instructions and the latency of the chain of divisions and table
// loads. (1M Gaussians, one fisheye camera: 96 -> 78 us, and 24M (camera, Gaussian)
// items 1810 -> 1470 us, with the SH rows copied 16 bytes a lane, one division per
// half-angle and the searches of arc_range.)
#ifndef GEER_PREP_MINB
#define GEER_PREP_MINB 3  // resident blocks per SM: caps registers at 80
#endif
// SPLAT: the instance for the association ablation and the splat alpha (any
// GEER_ASSOC_* / GEER_ALPHA_*); the PBF / exact-integral instance (SPLAT false)
// holds none of that code.
template <int DEG, bool SPLAT>
__global__ void __launch_bounds__(kPrepThreads, GEER_PREP_MINB) k_preprocess(
    const DevCam *__restrict__ cams, int ncams, const float4 *__restrict__ ttab, Params p,
    const float *__restrict__ mean, const float *__restrict__ scale, const float *__restrict__ quat,
    const float *__restrict__ opacity, const float *__restrict__ sh, int64_t n, Record *__restrict__ rec,
    uint4 *__restrict__ ranges, GradAcc *__restrict__ gacc, uint32_t *__restrict__ count, uint32_t *__restrict__ key,
    uint32_t *__restrict__ blocksum, int64_t nblk) {
    grid_dep_sync();
    constexpr int NC = ShRows<DEG>::NC, ST = ShRows<DEG>::kStride;
    extern __shared__ __align__(16) float s_sh[];  // [kPrepThreads][ST]
    const int64_t g0 = (int64_t)blockIdx.x * kPrepThreads;
    const int64_t g = g0 + threadIdx.x;
    {
        // the warp's SH coefficients, copied asynchronously while the bounds are
        // computed; read only for the colour
        const int w0 = threadIdx.x & ~31;
        const int rows = (int)min((int64_t)32, n - (g0 + w0));
        if (rows > 0) sh_stage<DEG>(s_sh + w0 * ST, sh + (g0 + w0) * NC, rows);
    }
    bool ok = g < n;
    float mu[3] = {0, 0, 0}, sc[3] = {1, 1, 1}, qt[4] = {1, 0, 0, 0}, sigma = 0.0f;
    if (ok) {
#pragma unroll
        for (int a = 0; a < 3; ++a) { mu[a] = mean[3 * g + a]; sc[a] = scale[3 * g + a]; }
#pragma unroll
        for (int a = 0; a < 4; ++a) qt[a] = quat[4 * g + a];
        sigma = opacity[g];
#pragma unroll
        for (int a = 0; a < 3; ++a)
            if (!isfinite(mu[a]) || !isfinite(sc[a]) || !(sc[a] > 0.0f)) ok = false;
#pragma unroll
        for (int a = 0; a < 4; ++a)
            if (!isfinite(qt[a])) ok = false;
        if (!isfinite(sigma) || !(sigma >= p.alpha_min)) ok = false;
    }
    // normalised quaternion and rotation, exactly rounded
    float R[9];
    float lam2 = 0.0f;
    if (ok) {
        float qn = fsq(fa(fa(fa(fm(qt[0], qt[0]), fm(qt[1], qt[1])), fm(qt[2], qt[2])), fm(qt[3], qt[3])));
        if (!(qn > 0.0f)) ok = false;
        float w = fdv(qt[0], qn), x = fdv(qt[1], qn), y = fdv(qt[2], qn), z = fdv(qt[3], qn);
        R[0] = fs(1.0f, fm(2.0f, fa(fm(y, y), fm(z, z))));
        R[1] = fm(2.0f, fs(fm(x, y), fm(w, z)));
        R[2] = fm(2.0f, fa(fm(x, z), fm(w, y)));
        R[3] = fm(2.0f, fa(fm(x, y), fm(w, z)));
        R[4] = fs(1.0f, fm(2.0f, fa(fm(x, x), fm(z, z))));
        R[5] = fm(2.0f, fs(fm(y, z), fm(w, x)));
        R[6] = fm(2.0f, fs(fm(x, z), fm(w, y)));
        R[7] = fm(2.0f, fa(fm(y, z), fm(w, x)));
        R[8] = fs(1.0f, fm(2.0f, fa(fm(x, x), fm(y, y))));
        lam2 = lambda2(sigma, p.alpha_min, p.lambda_pad);
        if (!(lam2 > 0.0f)) ok = false;
    }
    const float s2[3] = {fm(sc[0], sc[0]), fm(sc[1], sc[1]), fm(sc[2], sc[2])};
    const float ss[3] = {fm(sc[1], sc[2]), fm(sc[0], sc[2]), fm(sc[0], sc[1])};

    for (int ci = 0; ci < ncams; ++ci) {
        const DevCam &cam = cams[ci];
        const int64_t idx = (int64_t)ci * n + g;
        uint32_t cnt = 0;
        bool live = ok;
        float m0 = 0, m1 = 0, m2 = 0, M[9], u[3];
        Record r;
        if (live) {
            const float *Rc = cam.R;
            m0 = fa(fa(fa(fm(Rc[0], mu[0]), fm(Rc[1], mu[1])), fm(Rc[2], mu[2])), cam.t[0]);
            m1 = fa(fa(fa(fm(Rc[3], mu[0]), fm(Rc[4], mu[1])), fm(Rc[5], mu[2])), cam.t[1]);
            m2 = fa(fa(fa(fm(Rc[6], mu[0]), fm(Rc[7], mu[1])), fm(Rc[8], mu[2])), cam.t[2]);
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int j = 0; j < 3; ++j)
                    M[3 * i + j] = fa(fa(fm(Rc[3 * i], R[j]), fm(Rc[3 * i + 1], R[3 + j])), fm(Rc[3 * i + 2], R[6 + j]));
            // camera inside the lambda-ellipsoid: cull (App. B.2: t < 0 matters only
            // when the optical centre is inside the contour)
#pragma unroll
            for (int k = 0; k < 3; ++k)
                u[k] = fdv(fa(fa(fm(M[k], m0), fm(M[3 + k], m1)), fm(M[6 + k], m2)), sc[k]);
            float ou2 = fa(fa(fm(u[0], u[0]), fm(u[1], u[1])), fm(u[2], u[2]));
            if (!(ou2 > lam2)) live = false;
            // the splatting bounds and the splat alpha project through z: their near plane as well
            if (SPLAT && (p.assoc != GEER_ASSOC_PBF || p.alpha_model != GEER_ALPHA_EXACT) && !(m2 > kSplatNear))
                live = false;
        }
        float sp[5];  // GEER_ALPHA_SPLAT: the splat's centre and conic
        if (SPLAT && live && p.alpha_model != GEER_ALPHA_EXACT && !splat_conic(m0, m1, m2, M, sc, sp)) live = false;
        if (live) {
            Arc A, B, A1, B1;
            if (!SPLAT || p.assoc == GEER_ASSOC_PBF) {
                auto SIG = [&](int a, int b) {
                    return fa(fa(fm(s2[0], fm(M[3 * a], M[3 * b])), fm(s2[1], fm(M[3 * a + 1], M[3 * b + 1]))),
                              fm(s2[2], fm(M[3 * a + 2], M[3 * b + 2])));
                };
                float Sxx = SIG(0, 0), Syy = SIG(1, 1), Szz = SIG(2, 2), Sxz = SIG(0, 2), Syz = SIG(1, 2);
                float T00 = fs(fm(lam2, Sxx), fm(m0, m0));
                float T11 = fs(fm(lam2, Syy), fm(m1, m1));
                float T22 = fs(fm(lam2, Szz), fm(m2, m2));
                float T02 = fs(fm(lam2, Sxz), fm(m0, m2));
                float T12 = fs(fm(lam2, Syz), fm(m1, m2));
                float pxz[3], pyz[3], dxz[3], dyz[3];
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    float cx = fs(fm(m0, M[6 + k]), fm(m2, M[k]));
                    float cy = fs(fm(m1, M[6 + k]), fm(m2, M[3 + k]));
                    pxz[k] = fm(s2[k], fm(cx, cx));
                    pyz[k] = fm(s2[k], fm(cy, cy));
                    float ax = fm(ss[k], M[3 + k]);
                    float ay = fm(ss[k], M[k]);
                    dxz[k] = fm(ax, ax);
                    dyz[k] = fm(ay, ay);
                }
                float Pxz = fa(fa(pxz[0], pxz[1]), pxz[2]), Pyz = fa(fa(pyz[0], pyz[1]), pyz[2]);
                float Dxz = fa(fa(dxz[0], dxz[1]), dxz[2]), Dyz = fa(fa(dyz[0], dyz[1]), dyz[2]);
                A = pbf_arc(m0, m2, T00, T02, T22, Pxz, Dxz, lam2);
                B = pbf_arc(m1, m2, T11, T12, T22, Pyz, Dyz, lam2);
                A1 = shift_arc(A);
                B1 = shift_arc(B);
            } else {
                splat_arcs(p.assoc, p.snug, p.alpha_min, sigma, m0, m1, m2, M, sc, A, A1, B, B1);
            }
            const float4 *ctab = ttab + cam.tcol_off;
            const float4 *rtab = ttab + cam.trow_off;
            int rg[8] = {0, 0, 0, 0, 0, 0, 0, 0};
            const float chalf = 0.5f * (float)(cam.width - 1), rhalf = 0.5f * (float)(cam.height - 1);
            arc_range(A, ctab, cam.tiles_x, cam.col_ppr, chalf, rg[0], rg[1]);
            arc_range(B, rtab, cam.tiles_y, cam.row_ppr, rhalf, rg[4], rg[5]);
            if (cam.any_row_flip) arc_range(A1, ctab, cam.tiles_x, cam.col_ppr, chalf, rg[2], rg[3]);
            if (cam.any_col_flip) arc_range(B1, rtab, cam.tiles_y, cam.row_ppr, rhalf, rg[6], rg[7]);
            if (is_rect(cam, rg))
                cnt = (uint32_t)(rg[1] - rg[0]) * (uint32_t)(rg[5] - rg[4]);
            else
                cnt = assoc_count(cam, rg, 0, cam.tiles_x, 0, cam.tiles_y);
            float dist = fsq(fa(fa(fm(m0, m0), fm(m1, m1)), fm(m2, m2)));
            key[idx] = __float_as_uint(dist);
            ranges[idx] = make_uint4((uint32_t)rg[0] | ((uint32_t)rg[1] << 16), (uint32_t)rg[2] | ((uint32_t)rg[3] << 16),
                                     (uint32_t)rg[4] | ((uint32_t)rg[5] << 16), (uint32_t)rg[6] | ((uint32_t)rg[7] << 16));
            // render record: W = S^-1 M^T (camera frame), o_u = -W mu_c = -u; for the
            // splat alpha, W[0..4] = the splat's centre and conic instead
            if (!SPLAT || p.alpha_model == GEER_ALPHA_EXACT) {
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    float inv = 1.0f / sc[k];
                    r.W[3 * k + 0] = M[k] * inv;
                    r.W[3 * k + 1] = M[3 + k] * inv;
                    r.W[3 * k + 2] = M[6 + k] * inv;
                    r.ou[k] = -u[k];
                }
            } else {
#pragma unroll
                for (int k = 0; k < 9; ++k) r.W[k] = k < 5 ? sp[k] : 0.0f;
#pragma unroll
                for (int k = 0; k < 3; ++k) r.ou[k] = 0.0f;
            }
            r.log2_sigma = log2f(sigma);
        } else if (g < n) {
            key[idx] = 0u;
            ranges[idx] = make_uint4(0, 0, 0, 0);
        }
        if (ci == 0) {  // the warp's SH rows have arrived
            asm volatile("cp.async.wait_all;\n" ::: "memory");
            __syncwarp();
        }
        if (live) {
            float dx = mu[0] - cam.o[0], dy = mu[1] - cam.o[1], dz = mu[2] - cam.o[2];
            float inv = rsqrtf(dx * dx + dy * dy + dz * dz);
            sh_colour<DEG>(s_sh + threadIdx.x * ST, dx * inv, dy * inv, dz * inv, r.rgb);
            float4 *dst = reinterpret_cast<float4 *>(rec + idx);
            const float4 *src = reinterpret_cast<const float4 *>(&r);
#pragma unroll
            for (int i = 0; i < 4; ++i) dst[i] = src[i];
        }
        if (g < n) count[idx] = cnt;
        if (g < n && gacc) {  // every item's backward accumulators start from zero
            float4 *acc = reinterpret_cast<float4 *>(gacc + idx);
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
        const int tot = __syncthreads_count(cnt > 0);
        if (threadIdx.x == 0) blocksum[(int64_t)ci * nblk + blockIdx.x] = (uint32_t)tot;
    }
}

// The totals of a counting pass: pairs to sort (clamped to cap, with the capacity check).
__device__ __forceinline__ void put_pair_total(uint32_t *misc, unsigned long long total, int64_t cap) {
    misc[kMiscPairs] = (uint32_t)min(total, (unsigned long long)cap);
    misc[kMiscPairsHi] = (uint32_t)(total >> 32);
    misc[kMiscTotalLo] = (uint32_t)total;
    if (total > (unsigned long long)cap) atomicOr(&misc[kMiscStatus], kStatusCapacity);
}

// Exclusive scan of per-block counts (one block). mode 0 (live items): total -> misc[kMiscLive]; also clears the
// per-super-tile pair counts. mode 1 ((super-tile, item) pairs): total ->
// misc[kMiscPairs] (clamped to cap) with the capacity check. mode 2 ((tile, item)
// associations P): total -> misc[kMiscTileLo / Hi]. With two blocks, block 1
// scans blocksum_b in mode_b at the same time (one launch for two arrays).
__global__ void __launch_bounds__(1024) k_scan_blocks(uint32_t *__restrict__ blocksum, int64_t m,
                                                      uint32_t *__restrict__ misc, uint2 *__restrict__ srange,
                                                      int64_t nst, int64_t cap, int mode,
                                                      uint32_t *__restrict__ blocksum_b = nullptr, int mode_b = 0) {
    grid_dep_sync();
    __shared__ unsigned long long warp_tot[32];
    if (blockIdx.x == 1) {
        blocksum = blocksum_b;
        mode = mode_b;
    }
    if (mode != 0) m = ((int64_t)misc[kMiscLive] + kPrepThreads - 1) / kPrepThreads;  // the blocks with live items
    // 4096 counts at a time, four neighbouring ones a thread (one 16-byte access), with a running total
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    unsigned long long carry = 0;
    const auto load = [&](int64_t i) {
        if (i + 4 <= m) return *reinterpret_cast<const uint4 *>(blocksum + i);
        return make_uint4(i < m ? blocksum[i] : 0u, i + 1 < m ? blocksum[i + 1] : 0u, i + 2 < m ? blocksum[i + 2] : 0u, 0u);
    };
    uint4 c = load(4 * t);
    for (int64_t i0 = 0; i0 < m; i0 += 4096) {
        const int64_t i = i0 + 4 * t;
        const uint4 next = i0 + 4096 < m ? load(i + 4096) : make_uint4(0u, 0u, 0u, 0u);
        const unsigned long long s = (unsigned long long)c.x + c.y + c.z + c.w;
        unsigned long long v = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            unsigned long long y = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += y;
        }
        if (lane == 31) warp_tot[warp] = v;
        __syncthreads();
        unsigned long long w = warp_tot[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            unsigned long long y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        const unsigned long long before = __shfl_sync(0xffffffffu, w, max(warp - 1, 0));
        unsigned long long excl = carry + v - s + (warp > 0 ? before : 0ull);
        carry += __shfl_sync(0xffffffffu, w, 31);
        __syncthreads();
        uint4 o4;
        const auto put = [&](uint32_t n) {
            const uint32_t e = (uint32_t)min(excl, 0xffffffffull);
            excl += n;
            return e;
        };
        o4.x = put(c.x);
        o4.y = put(c.y);
        o4.z = put(c.z);
        o4.w = put(c.w);
        if (i + 4 <= m) {
            *reinterpret_cast<uint4 *>(blocksum + i) = o4;
        } else {
            if (i < m) blocksum[i] = o4.x;
            if (i + 1 < m) blocksum[i + 1] = o4.y;
            if (i + 2 < m) blocksum[i + 2] = o4.z;
        }
        c = next;
    }
    if (t == 0) {
        const unsigned long long total = carry;
        if (mode == 0) {
            misc[kMiscLive] = (uint32_t)total;
            // the depth sort's first pass reads buffer 0 (see depth_sorted_buf)
            misc[kMiscSortCur] = 1u;
            misc[kMiscSortSame] = 0u;
        } else if (mode == 2) {
            misc[kMiscTileLo] = (uint32_t)total;
            misc[kMiscTileHi] = (uint32_t)(total >> 32);
        } else {
            put_pair_total(misc, total, cap);
        }
    }
    if (mode == 0) {
        uint32_t *scount = reinterpret_cast<uint32_t *>(srange + nst);
        for (int64_t i = t; i < nst; i += 1024) scount[i] = 0u;
    }
}

// Compaction of the live (camera, Gaussian) items, in index order, into
// (depth key, item) arrays. Block (b, ci): the Gaussians of kCompact preprocess blocks
// of camera ci, all loads in flight together.
constexpr int kCompact = 4;
__global__ void __launch_bounds__(kPrepThreads) k_compact(int64_t n, const uint32_t *__restrict__ count,
                                                          const uint32_t *__restrict__ key,
                                                          const uint32_t *__restrict__ blocksum, int64_t nblk,
                                                          uint32_t *__restrict__ okey, uint32_t *__restrict__ oid) {
    grid_dep_sync();
    __shared__ uint32_t s_wsum[kCompact][kPrepThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t b0 = (int64_t)blockIdx.x * kCompact, i0 = (int64_t)blockIdx.y * n;
    uint32_t k[kCompact], pos[kCompact], live[kCompact];
#pragma unroll
    for (int u = 0; u < kCompact; ++u) {
        const int64_t g = (b0 + u) * kPrepThreads + threadIdx.x;
        const bool in = g < n;
        const bool on = in && count[i0 + g] > 0;
        k[u] = in ? key[i0 + g] : 0u;
        pos[u] = b0 + u < nblk ? blocksum[(int64_t)blockIdx.y * nblk + b0 + u] : 0u;
        live[u] = __ballot_sync(0xffffffffu, on);
        if (lane == 0) s_wsum[u][warp] = (uint32_t)__popc(live[u]);
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kCompact; ++u) {
        for (int w = 0; w < warp; ++w) pos[u] += s_wsum[u][w];
        if (live[u] >> lane & 1u) {
            const uint32_t p = pos[u] + (uint32_t)__popc(live[u] & ((1u << lane) - 1u));
            okey[p] = k[u];
            oid[p] = (uint32_t)(i0 + (b0 + u) * kPrepThreads + threadIdx.x);
        }
    }
}

// x / S for a tile index x, inv_s = super_inverse(S): exact for S < 9 and x < 2^28.
__device__ __forceinline__ uint32_t super_inverse(int S) { return S > 1 ? 0xffffffffu / (uint32_t)S + 1u : 0u; }
__device__ __forceinline__ int super_of(int x, uint32_t inv_s) {
    return inv_s ? (int)__umulhi((uint32_t)x, inv_s) : x;
}

// A live item's association for the binning: its only rectangle (packed columns
// and rows, lo | hi << 16) when it is one (rects 1: all but the Gaussians across a
// tile column or row where the other angle passes 90 degrees).
struct Assoc {
    uint32_t xr, yr, rects;
};

__device__ __forceinline__ Assoc item_assoc(const DevCam &cam, const uint4 r4) {
    Assoc a{r4.x, r4.z, 1u};
    int rg[8];
    unpack_ranges(r4, rg);
    if (!is_rect(cam, rg)) {
        a.rects = 0;
        assoc_rects(cam, rg, [&](int4 r) {
            a.xr = (uint32_t)r.x | (uint32_t)r.y << 16;
            a.yr = (uint32_t)r.z | (uint32_t)r.w << 16;
            ++a.rects;
        });
    }
    return a;
}

// The super-tile box of a rectangle: first column and row, columns, super-tiles.
struct SuperBox {
    int sx0, sy0, w;
    uint32_t supers;
};
__device__ __forceinline__ SuperBox super_box(uint32_t xr, uint32_t yr, uint32_t inv_s) {
    SuperBox b;
    b.sx0 = super_of((int)(xr & 0xffff), inv_s);
    b.sy0 = super_of((int)(yr & 0xffff), inv_s);
    b.w = super_of((int)(xr >> 16) - 1, inv_s) + 1 - b.sx0;
    b.supers = (uint32_t)(b.w * (super_of((int)(yr >> 16) - 1, inv_s) + 1 - b.sy0));
    return b;
}

// The super-tiles of an item of several rectangles, by one thread: the union of the
// rectangles' super-tile boxes, each super-tile once, while the boxes hold at most
// kThreadCells super-tiles; else nothing is done and false returned.
constexpr uint32_t kThreadCells = 6;
template <typename F>
__device__ __forceinline__ bool thread_supers(const DevCam &cam, uint32_t inv_s, const uint4 r4, F f) {
    int rg[8];
    unpack_ranges(r4, rg);
    int4 box[9];
    int n = 0;
    uint32_t cells = 0;
    assoc_rects(cam, rg, [&](int4 r) {
        const int4 b = make_int4(super_of(r.x, inv_s), super_of(r.y - 1, inv_s), super_of(r.z, inv_s),
                                 super_of(r.w - 1, inv_s));
        cells += (uint32_t)((b.y - b.x + 1) * (b.w - b.z + 1));
        box[n++] = b;
    });
    if (cells > kThreadCells) return false;
    for (int k = 0; k < n; ++k)
        for (int sy = box[k].z; sy <= box[k].w; ++sy)
            for (int sx = box[k].x; sx <= box[k].y; ++sx) {
                bool seen = false;
                for (int q = 0; q < k && !seen; ++q)
                    seen = sx >= box[q].x && sx <= box[q].y && sy >= box[q].z && sy <= box[q].w;
                if (!seen) f(sx, sy, rg);
            }
    return true;
}

// Bits [lo, hi) of the S tile columns (or rows) that start at base.
__device__ __forceinline__ uint32_t span_bits(int lo, int hi, int base, int S) {
    const int l = min(max(lo - base, 0), S), h = min(max(hi - base, 0), S);
    return h > l ? (1u << h) - (1u << l) : 0u;
}

// An item's association within super-tiles as four sets of tile columns times sets of
// tile rows. A tile (x, y) is associated when (x in X0 and row y has rays with cos(phi)
// >= 0, or x in X1 and row y has rays with cos(phi) <= 0), and likewise for its row in
// Y0 / Y1 with the column's flags; multiplied out, byte k of super_cols (the columns of
// super-tile column sx) goes with byte k of super_rows (the rows of super-tile row sy).
__device__ __forceinline__ uint32_t super_cols(const DevCam &cam, const int rg[8], int sx, int S) {
    const int x0 = sx * S;
    const uint32_t X0 = span_bits(rg[0], rg[1], x0, S), X1 = span_bits(rg[2], rg[3], x0, S);
    const uint32_t z = span_bits(cam.zc[0], cam.zc[1], x0, S);
    const uint32_t w = span_bits(0, cam.wc[0], x0, S) | span_bits(cam.wc[1], cam.tiles_x, x0, S);
    return (X0 & z) | (X0 & w) << 8 | (X1 & z) << 16 | (X1 & w) << 24;
}
__device__ __forceinline__ uint32_t super_rows(const DevCam &cam, const int rg[8], int sy, int S) {
    const int y0 = sy * S;
    const uint32_t Y0 = span_bits(rg[4], rg[5], y0, S), Y1 = span_bits(rg[6], rg[7], y0, S);
    const uint32_t z = span_bits(cam.zr[0], cam.zr[1], y0, S);
    const uint32_t w = span_bits(0, cam.wr[0], y0, S) | span_bits(cam.wr[1], cam.tiles_y, y0, S);
    return (Y0 & z) | (Y1 & z) << 8 | (Y0 & w) << 16 | (Y1 & w) << 24;
}

// The super-tile columns (or rows) that hold the tiles [a0, a1) and [b0, b1).
__device__ __forceinline__ int2 super_span(int a0, int a1, int b0, int b1, uint32_t inv_s) {
    const bool a = a0 < a1, b = b0 < b1;
    if (!a && !b) return make_int2(0, 0);
    return make_int2(super_of(min(a ? a0 : b0, b ? b0 : a0), inv_s), super_of(max(a ? a1 : b1, b ? b1 : a1) - 1, inv_s) + 1);
}

// The number of super-tiles of an item (rg the same in every lane), by its warp: a lane
// per super-tile column, whose sets that are not empty become bits of four words, then a
// lane per row.
__device__ __forceinline__ uint32_t warp_super_count(const DevCam &cam, const int rg[8], int S, uint32_t inv_s) {
    const int lane = threadIdx.x & 31;
    const int2 xs = super_span(rg[0], rg[1], rg[2], rg[3], inv_s), ys = super_span(rg[4], rg[5], rg[6], rg[7], inv_s);
    uint32_t n = 0;
    for (int x0 = xs.x; x0 < xs.y; x0 += 32) {
        const uint32_t c = super_cols(cam, rg, x0 + lane, S);  // (columns past the image are empty)
        uint32_t on[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) on[k] = __ballot_sync(0xffffffffu, c >> (8 * k) & 0xffu);
        for (int y0 = ys.x; y0 < ys.y; y0 += 32) {
            const uint32_t r = super_rows(cam, rg, y0 + lane, S);
            uint32_t any = 0;
#pragma unroll
            for (int k = 0; k < 4; ++k) any |= r >> (8 * k) & 0xffu ? on[k] : 0u;
            n += (uint32_t)__popc(any);
        }
    }
    return __reduce_add_sync(0xffffffffu, n);
}

// One item a lane (live: whether it has one): its rectangle and number of super-tiles,
// and its tiles.
struct ItemPairs {
    uint32_t xr, yr, supers, tiles;  // xr 0: several rectangles
};
__device__ __forceinline__ ItemPairs warp_item_pairs(const DevCam *__restrict__ cams, int S, uint32_t inv_s, bool live,
                                                     int ci, const uint4 r4) {
    const int lane = threadIdx.x & 31;
    Assoc a{0u, 0u, 0u};
    ItemPairs p{0u, 0u, 0u, 0u};
    if (live) a = item_assoc(cams[ci], r4);
    if (a.rects == 1) {
        p.xr = a.xr;
        p.yr = a.yr;
        p.supers = super_box(a.xr, a.yr, inv_s).supers;
        p.tiles = ((a.xr >> 16) - (a.xr & 0xffff)) * ((a.yr >> 16) - (a.yr & 0xffff));
    }
    // items of several rectangles: those of few super-tiles by their threads, the others by
    // the warp one at a time, with a lane per super-tile column and row. (Preprocess and
    // binning of 1M Gaussians of a room around a 190 degree camera, 15% of them of several
    // rectangles, with threads up to 0 / 6 / 16 / 64 super-tiles: 277 / 270 / 273 / 313 us;
    // 358 with a lane per super-tile of every rectangle's box, each tested against the
    // boxes before. 1M on a shell at 205 degrees: 312 / 214 / 214 / 217, 219 with boxes.)
    bool by_warp = false;
    if (a.rects > 1) {
        const DevCam &cam = cams[ci];
        by_warp = !thread_supers(cam, inv_s, r4, [&](int, int, const int *) { ++p.supers; });
        int rg[8];
        unpack_ranges(r4, rg);
        p.tiles = assoc_count(cam, rg, 0, cam.tiles_x, 0, cam.tiles_y);
    }
    for (uint32_t many = __ballot_sync(0xffffffffu, by_warp); many; many &= many - 1) {
        const int o = __ffs(many) - 1;
        const uint4 q = make_uint4(__shfl_sync(0xffffffffu, r4.x, o), __shfl_sync(0xffffffffu, r4.y, o),
                                   __shfl_sync(0xffffffffu, r4.z, o), __shfl_sync(0xffffffffu, r4.w, o));
        int rg[8];
        unpack_ranges(q, rg);
        const uint32_t k = warp_super_count(cams[__shfl_sync(0xffffffffu, ci, o)], rg, S, inv_s);
        if (lane == o) p.supers = k;
    }
    return p;
}

// Per 256 depth-sorted live items (a block of the emission): their super-tile pairs
// (emission offsets) and their tile pairs (the total, for the capacity check). Each
// item's rectangle and super-tiles are left in depth order for the emission, in the
// depth sort's buffers, which nobody reads any more: columns and rows in the keys'
// (columns 0: several rectangles), super-tiles in the unused ids'. Bound by the
// scattered reads of the items' ranges: the tile counts follow from them (a second
// scattered read took as long), and a thread has kGather items in flight.
constexpr int kGather = 2;  // (24M items, 9M live: 273 us; with 1 320, with 4 299; both arrays read 452)
__global__ void __launch_bounds__(kPrepThreads) k_gather_counts(
    const DevCam *__restrict__ cams, int64_t n, int S, uint32_t *__restrict__ id0, uint32_t *__restrict__ id1,
    const uint4 *__restrict__ ranges, const uint32_t *__restrict__ misc, uint32_t *__restrict__ bs_super,
    uint32_t *__restrict__ bs_tile, uint32_t *__restrict__ oxr, uint32_t *__restrict__ oyr) {
    grid_dep_sync();
    __shared__ uint32_t s_sum[kGather][2];
    const uint32_t L = misc[kMiscLive];
    const int64_t i0 = (int64_t)blockIdx.x * (kGather * kPrepThreads);
    if (i0 >= L) return;
    const bool cur = depth_sorted_buf(misc) != 0;
    const uint32_t *__restrict__ sorted_id = cur ? id1 : id0;
    uint32_t *__restrict__ osupers = cur ? id0 : id1;
    const int lane = threadIdx.x & 31;
    const uint32_t inv_s = super_inverse(S);
    if (threadIdx.x < 2 * kGather) (&s_sum[0][0])[threadIdx.x] = 0u;
    uint32_t item[kGather];
    uint4 r4[kGather];
#pragma unroll
    for (int u = 0; u < kGather; ++u) {
        const int64_t i = i0 + u * kPrepThreads + threadIdx.x;
        item[u] = i < L ? sorted_id[i] : 0u;
    }
#pragma unroll
    for (int u = 0; u < kGather; ++u) {
        r4[u] = make_uint4(0u, 0u, 0u, 0u);
        if (i0 + u * kPrepThreads + threadIdx.x < L) r4[u] = ranges[item[u]];
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kGather; ++u) {
        const int64_t i = i0 + u * kPrepThreads + threadIdx.x;
        const ItemPairs p = warp_item_pairs(cams, S, inv_s, i < L, (int)(item[u] / (uint32_t)n), r4[u]);
        if (i < L) {
            oxr[i] = p.xr;
            oyr[i] = p.yr;
            osupers[i] = p.supers;
        }
        const uint32_t tiles = __reduce_add_sync(0xffffffffu, p.tiles), supers = __reduce_add_sync(0xffffffffu, p.supers);
        if (lane == 0) {
            atomicAdd(&s_sum[u][0], supers);
            atomicAdd(&s_sum[u][1], tiles);
        }
    }
    __syncthreads();
    if (threadIdx.x < kGather && i0 + threadIdx.x * kPrepThreads < L) {
        bs_super[(int64_t)blockIdx.x * kGather + threadIdx.x] = s_sum[threadIdx.x][0];
        bs_tile[(int64_t)blockIdx.x * kGather + threadIdx.x] = s_sum[threadIdx.x][1];
    }
}

// Everything between the preprocess and the emission for at most kClusterItems (camera,
// Gaussian) items, in one block or in a cluster of C: compaction, the stable depth sort
// (8-bit digits, the keys and ids held in registers through a pass and reordered in
// shared memory; a pass whose digit all keys share is skipped), the counting in depth
// order and the scans. It leaves what those kernels leave (ids in buffer 0). In a
// cluster each block holds an equal part of the order, the digits' totals are read from
// and the keys written to the other blocks' shared memory. One block is bound by the
// issue rate of its SM, the cluster by its two barriers a pass; the twelve launches
// replaced take about 4 us each at these sizes, whatever their work. Preprocess to
// render order, one block / cluster / launches: 2048 items 41 / - / 67 us, 4096
// 45 / - / 71, 6000 51 / 50 / 73, 8192 57 / 51 / 69, 12001 78 / 56 / 73, 20000 - / 63 /
// 73, 32768 - / 73 / 75: hence the lines. (The lanes of a digit by a vote per bit instead
// of shared masks: 60 at 8192; by __match_any_sync: 71.) K: items a thread.
constexpr int kSmallItems = 4096, kClusterItems = 32768, kSmallThreads = 1024, kCluster = 8;
template <int K, int C>
__global__ void __launch_bounds__(kSmallThreads) k_small_front(
    const DevCam *__restrict__ cams, int64_t n, int items, int S, const uint32_t *__restrict__ count,
    const uint32_t *__restrict__ key, const uint4 *__restrict__ ranges, uint32_t *__restrict__ misc,
    uint32_t *__restrict__ id0, uint32_t *__restrict__ id1, uint32_t *__restrict__ oxr, uint32_t *__restrict__ oyr,
    uint32_t *__restrict__ bs_super, uint32_t *__restrict__ scount, int64_t nst, int64_t cap) {
    grid_dep_sync();
    constexpr int W = kSmallThreads / 32, CHUNKS = K * kSmallThreads / kPrepThreads;
    extern __shared__ uint32_t dyn[];
    uint32_t(*s_hist)[kRadix] = reinterpret_cast<uint32_t(*)[kRadix]>(dyn);  // [W]: a warp's keys per digit
    uint32_t(*s_match)[kRadix] = s_hist + W;  // lane masks per digit, zero between ranking steps
    uint32_t *s_key = dyn + 2 * W * kRadix;   // [K * kSmallThreads]
    uint16_t *s_val = reinterpret_cast<uint16_t *>(s_key + K * kSmallThreads);
    __shared__ uint32_t s_part[kSmallThreads / kRadix][kRadix];
    __shared__ uint32_t s_wsum[W];
    __shared__ uint32_t s_sum[CHUNKS][2];
    // what the other blocks of the cluster read: live items, digit totals (two passes' in turn), pairs and tiles
    __shared__ uint32_t s_live, s_dig[C > 1 ? 2 : 1][kRadix], s_low[kSmallThreads / kRadix][C > 1 ? kRadix : 1];
    __shared__ unsigned long long s_total[2];
    const auto cluster = cooperative_groups::this_cluster();
    const int cta = C > 1 ? (int)cluster.block_rank() : 0;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const uint32_t below = (1u << lane) - 1u;
    for (int64_t i = cta * kSmallThreads + t; i < nst; i += C * kSmallThreads) scount[i] = 0u;
    for (int i = t; i < W * kRadix; i += kSmallThreads) (&s_match[0][0])[i] = 0u;
    for (int i = t; i < 2 * CHUNKS; i += kSmallThreads) (&s_sum[0][0])[i] = 0u;
    // compaction in index order: a warp's 32 K consecutive items
    uint32_t kk[K], live[K], mine = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int i = ((cta * W + warp) * K + k) * 32 + lane;
        const bool on = i < items && count[i] > 0u;
        kk[k] = i < items ? key[i] : 0u;
        live[k] = __ballot_sync(0xffffffffu, on);
        mine += (uint32_t)__popc(live[k]);
    }
    if (lane == 0) s_wsum[warp] = mine;
    __syncthreads();
    uint32_t v = s_wsum[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
    }
    int L = (int)__shfl_sync(0xffffffffu, v, 31);
    uint32_t at = warp ? __shfl_sync(0xffffffffu, v, max(warp - 1, 0)) : 0u;
    // C > 1: block c holds the places [c per, (c + 1) per) of the order
    int per = K * kSmallThreads, own = L;
    if constexpr (C > 1) {
        if (t == 0) s_live = (uint32_t)L;
        cluster.sync();
        L = 0;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const int x = (int)*cluster.map_shared_rank(&s_live, c);
            at += c < cta ? x : 0;
            L += x;
        }
        per = max((L + C * kPrepThreads - 1) / (C * kPrepThreads), 1) * kPrepThreads;
        own = min(max(L - cta * per, 0), per);
    }
    const auto put = [&](uint32_t pos, uint32_t k, uint32_t val) {
        if constexpr (C > 1) {
            const int c = (int)pos / per, e = (int)pos - c * per;
            cluster.map_shared_rank(s_key, c)[e] = k;
            cluster.map_shared_rank(s_val, c)[e] = (uint16_t)val;
        } else {
            s_key[pos] = k;
            s_val[pos] = (uint16_t)val;
        }
    };
    const auto sync_all = [&] {
        if constexpr (C > 1) cluster.sync();
        else __syncthreads();
    };
#pragma unroll
    for (int k = 0; k < K; ++k) {
        if (live[k] >> lane & 1u) {
            put(at + (uint32_t)__popc(live[k] & below), kk[k], (uint32_t)(((cta * W + warp) * K + k) * 32 + lane));
        }
        at += (uint32_t)__popc(live[k]);
    }
    sync_all();
    // the sort: a warp takes 32 kr consecutive keys
    const int kr = ((C > 1 ? per : L) + kSmallThreads - 1) / kSmallThreads;
#pragma unroll 1
    for (int shift = 0; shift < 32; shift += kRadixBits) {
        uint32_t val[K], rank[K];
        const uint32_t d0 = own > 0 ? (s_key[0] >> shift) & 0xffu : 0u;
        bool same = true;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int e = (warp * kr + k) * 32 + lane;
            if (k < kr && e < own) {
                kk[k] = s_key[e];
                val[k] = s_val[e];
                same = same && ((kk[k] >> shift) & 0xffu) == d0;
            }
        }
        for (int i = t; i < W * kRadix; i += kSmallThreads) (&s_hist[0][0])[i] = 0u;
        if (__syncthreads_and(same) && C == 1) continue;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            if (k >= kr) break;
            const bool on = (warp * kr + k) * 32 + lane < own;
            const uint32_t d = on ? (kk[k] >> shift) & 0xffu : 0u;
            if (on) atomicOr(&s_match[warp][d], 1u << lane);
            const uint32_t b = s_hist[warp][d];
            __syncwarp();
            const uint32_t peers = s_match[warp][d], before = (uint32_t)__popc(peers & below);
            __syncwarp();
            if (on && before == 0) {
                s_hist[warp][d] = b + (uint32_t)__popc(peers);
                s_match[warp][d] = 0u;
            }
            rank[k] = b + before;
            __syncwarp();
        }
        __syncthreads();
        // per digit the warps' places: a thread scans eight warps of one digit
        constexpr int Q = W / (kSmallThreads / kRadix);
        const int d = t & (kRadix - 1), q = t / kRadix;
        uint32_t c[Q], sum = 0;
#pragma unroll
        for (int w = 0; w < Q; ++w) {
            c[w] = s_hist[q * Q + w][d];
            sum += c[w];
        }
        s_part[q][d] = sum;
        __syncthreads();
        uint32_t pre = 0, tot = 0;
#pragma unroll
        for (int p = 0; p < kSmallThreads / kRadix; ++p) {
            const uint32_t x = s_part[p][d];
            pre += p < q ? x : 0u;
            tot += x;
        }
        if constexpr (C > 1) {
            // the blocks' totals of the digit; a quarter of this block reads a quarter of them
            static_assert(C == 2 * (kSmallThreads / kRadix), "two blocks a quarter");
            uint32_t *dig = s_dig[shift / kRadixBits & 1];
            if (q == 0) dig[d] = tot;
            cluster.sync();
            const uint32_t x0 = cluster.map_shared_rank(dig, 2 * q)[d], x1 = cluster.map_shared_rank(dig, 2 * q + 1)[d];
            s_part[q][d] = x0 + x1;
            s_low[q][d] = (2 * q < cta ? x0 : 0u) + (2 * q + 1 < cta ? x1 : 0u);
            __syncthreads();
            tot = 0;
#pragma unroll
            for (int p = 0; p < kSmallThreads / kRadix; ++p) {
                tot += s_part[p][d];
                pre += s_low[p][d];
            }
            if (__syncthreads_or(tot == (uint32_t)L)) continue;  // (in every block alike)
        }
        uint32_t sc = tot;  // scan over the digits (each quarter of the block the same)
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, sc, o);
            if (lane >= o) sc += y;
        }
        if (lane == 31) s_wsum[warp] = sc;
        __syncthreads();
        uint32_t run = sc - tot + pre;
#pragma unroll
        for (int w = 0; w < kRadix / 32; ++w) run += w < (warp & (kRadix / 32 - 1)) ? s_wsum[w] : 0u;
#pragma unroll
        for (int w = 0; w < Q; ++w) {
            s_hist[q * Q + w][d] = run;
            run += c[w];
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (k < kr && (warp * kr + k) * 32 + lane < own)
                put(s_hist[warp][(kk[k] >> shift) & 0xffu] + rank[k], kk[k], val[k]);
        sync_all();
    }
    // the counting, in depth order
    const uint32_t inv_s = super_inverse(S);
    for (int e0 = 0; e0 < own; e0 += kSmallThreads) {
        const int e = e0 + t, i = cta * per + e;
        const bool on = e < own;
        const uint32_t item = on ? s_val[e] : 0u;
        const uint4 r4 = on ? ranges[item] : make_uint4(0u, 0u, 0u, 0u);
        const ItemPairs p = warp_item_pairs(cams, S, inv_s, on, (int)(item / (uint32_t)n), r4);
        if (on) {
            id0[i] = item;
            oxr[i] = p.xr;
            oyr[i] = p.yr;
            id1[i] = p.supers;
        }
        const uint32_t tiles = __reduce_add_sync(0xffffffffu, p.tiles), supers = __reduce_add_sync(0xffffffffu, p.supers);
        if (lane == 0) {
            atomicAdd(&s_sum[e / kPrepThreads][0], supers);
            atomicAdd(&s_sum[e / kPrepThreads][1], tiles);
        }
    }
    if (t < 2) s_total[t] = 0ull;
    __syncthreads();
    if (t < 2 * CHUNKS) atomicAdd(&s_total[t & 1], (unsigned long long)s_sum[t >> 1][t & 1]);
    sync_all();
    unsigned long long pairs = 0, all_pairs = 0, all_tiles = 0;  // pairs: of the blocks before
#pragma unroll
    for (int c = 0; c < C; ++c) {
        const unsigned long long *x = C > 1 ? cluster.map_shared_rank(s_total, c) : s_total;
        pairs += c < cta ? x[0] : 0ull;
        all_pairs += x[0];
        all_tiles += x[1];
    }
    if constexpr (C > 1) cluster.sync();  // a block's shared memory is read until here
    if (warp > 0) return;
    for (int c0 = 0; c0 < CHUNKS; c0 += 32) {
        const uint32_t a = c0 + lane < CHUNKS ? s_sum[c0 + lane][0] : 0u;
        unsigned long long x = a;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long u = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += u;
        }
        if ((c0 + lane) * kPrepThreads < own)
            bs_super[cta * per / kPrepThreads + c0 + lane] = (uint32_t)min(pairs + x - a, 0xffffffffull);
        pairs += __shfl_sync(0xffffffffu, x, 31);
    }
    if (cta == 0 && lane == 0) {
        misc[kMiscLive] = (uint32_t)L;
        misc[kMiscSortCur] = 1u;  // the sorted ids are in buffer 0 (depth_sorted_buf)
        misc[kMiscSortSame] = 0u;
        misc[kMiscTileLo] = (uint32_t)all_tiles;
        misc[kMiscTileHi] = (uint32_t)(all_tiles >> 32);
        put_pair_total(misc, all_pairs, cap);
    }
}

// The tile mask of an item and super-tile: bit j * S + i for its tile (sx S + i, sy S + j).
// cols, rows: super_cols, super_rows; spread[r]: bit j * S for every bit j of r.
template <typename M>
__device__ __forceinline__ M tile_mask_sets(uint32_t cols, uint32_t rows, const M *spread) {
    M m = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) m |= spread[rows >> (8 * k) & 0xffu] * (M)(cols >> (8 * k) & 0xffu);
    return m;
}

// The same for a rectangle that meets the super-tile: columns [xlo, xhi) x rows
// [ylo, yhi) (packed lo | hi << 16). M: uint32_t where the S * S bits fit it.
template <typename M>
__device__ __forceinline__ M tile_mask_rect(uint32_t xr, uint32_t yr, int sx, int sy, int S, const M *spread) {
    const int x0 = sx * S, y0 = sy * S;
    const int xl = max((int)(xr & 0xffff) - x0, 0), xh = min((int)(xr >> 16) - x0, S);
    const int yl = max((int)(yr & 0xffff) - y0, 0), yh = min((int)(yr >> 16) - y0, S);
    return spread[(1u << yh) - (1u << yl)] * (M)((1u << xh) - (1u << xl));
}

__device__ __forceinline__ void put_mask(uint32_t *out, uint32_t i, uint32_t m) { out[i] = m; }
__device__ __forceinline__ void put_mask(uint32_t *out, uint32_t i, uint64_t m) {
    reinterpret_cast<uint2 *>(out)[i] = make_uint2((uint32_t)m, (uint32_t)(m >> 32));
}

// DuplicateWithKeys in depth order, at super-tile granularity: item i of the
// depth-sorted list emits one (global super-tile, item) pair per super-tile
// holding an associated tile, with its tile mask (what the renders' list fills
// test: one bit of a 4-byte load, where the 16 bytes of ranges cost an unpacking and
// eight comparisons), and counts the pairs per super-tile. An item's pairs may come
// in any order (each belongs to another super-tile). Items whose association is one
// rectangle are emitted by the whole warp together (lane j writes output j:
// coalesced) from a list in shared memory; the few others by the warp one by one (a
// thread looping over its item's super-tiles kept its block waiting). At most the
// resident blocks go through the items and add their counts to the global ones at the
// end: a block per 256 items added 8M for 12M pairs on 3600 super-tiles, 149 us where
// this takes 115 (with twice the blocks 116; 1M-Gaussian fisheye 30 -> 24).
// M: the mask's type (32 bits up to S = 5).
template <typename M>
__global__ void __launch_bounds__(kPrepThreads) k_duplicate(
    const DevCam *__restrict__ cams, int64_t n, int S, const uint32_t *__restrict__ id0,
    const uint32_t *__restrict__ id1, const uint32_t *__restrict__ xrs, const uint32_t *__restrict__ yrs,
    const uint4 *__restrict__ ranges, uint32_t *__restrict__ misc, const uint32_t *__restrict__ blocksum,
    uint32_t *__restrict__ okeys, uint32_t *__restrict__ ovals, uint32_t *__restrict__ omask,
    uint32_t *__restrict__ scount, int nst, int64_t cap) {
    grid_dep_sync();
    // a one-rectangle item: {columns, rows, item, first output (of the block's)},
    // {first output (of the warp's), super-tiles a row | stiles_x << 16, first super-tile, its x | y << 16}
    __shared__ uint4 s_item[kPrepThreads][2];
    __shared__ uint32_t wsum[kPrepThreads / 32];
    __shared__ uint2 s_sets[kPrepThreads / 32][32];          // a warp's super_cols and super_rows
    __shared__ M s_spread[sizeof(M) == 4 ? 32 : kPrepThreads];  // (S <= 5, S <= 8)
    extern __shared__ uint32_t sh[];  // per-super-tile pair counts when they fit (nst <= kSmemTiles)
    const bool smem = nst <= kSmemTiles;
    const uint32_t L = misc[kMiscLive];
    if ((int64_t)blockIdx.x * kPrepThreads >= L) return;
    if (smem)
        for (int k = threadIdx.x; k < nst; k += kPrepThreads) sh[k] = 0u;
    if (threadIdx.x < 1u << S) {
        M m = 0;
        for (int j = 0; j < S; ++j) m |= (M)(threadIdx.x >> j & 1u) << (j * S);
        s_spread[threadIdx.x] = m;
    }
    const auto count = [&](uint32_t st) {
        if (!in_bounds(st, (uint64_t)nst, kSiteDupSuper, misc)) return;
        if (smem) atomicAdd(&sh[st], 1u);
        else atomicAdd(&scount[st], 1u);
    };
    const bool cur = depth_sorted_buf(misc) != 0;
    const int lane = threadIdx.x & 31;
    const uint32_t inv_s = super_inverse(S);
    for (int64_t chunk = blockIdx.x; chunk * kPrepThreads < L; chunk += gridDim.x) {
        const int64_t i = chunk * kPrepThreads + threadIdx.x;
        uint32_t item = 0, xr = 0, yr = 0, cnt = 0;  // as the counting left them
        if (i < L) {
            item = (cur ? id1 : id0)[i];
            cnt = (cur ? id0 : id1)[i];
            xr = xrs[i];
            yr = yrs[i];
        }
        const int ci = (int)(item / (uint32_t)n);
        const DevCam &cam = cams[ci];
        uint32_t tot;
        const uint32_t pre = block_excl_scan(cnt, wsum, tot);  // (its barriers also follow the clearing of sh)
        const uint32_t base = blocksum[chunk];  // (pairs that fit have 32-bit places: cap < 2^32)
        const bool fits = (int64_t)base + pre + cnt <= cap;
        // cooperative emission of the warp's one-rectangle items
        const bool one = xr != 0 && fits;
        const uint32_t rc = one ? cnt : 0u;
        uint32_t incl = rc;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        const uint32_t ones = __ballot_sync(0xffffffffu, one);
        uint4(*list)[2] = s_item + (threadIdx.x & ~31);
        if (one) {
            const SuperBox b = super_box(xr, yr, inv_s);
            const int k = __popc(ones & ((1u << lane) - 1u));
            list[k][0] = make_uint4(xr, yr, item, pre);
            list[k][1] = make_uint4(incl - rc, (uint32_t)b.w | (uint32_t)cam.stiles_x << 16,
                                    (uint32_t)(cam.stile_base + b.sy0 * cam.stiles_x + b.sx0),
                                    (uint32_t)b.sx0 | (uint32_t)b.sy0 << 16);
        }
        __syncwarp();
        const uint32_t wtot = __shfl_sync(0xffffffffu, incl, 31);
        int before = -1;  // items that start in the windows so far, less one
        for (uint32_t j0 = 0; j0 < wtot; j0 += 32) {
            // the outputs of this window where an item starts; an output's item is the last to start
            const uint32_t at = incl - rc - j0;
            const uint32_t starts = __reduce_or_sync(0xffffffffu, one && at < 32u ? 1u << at : 0u);
            const uint32_t j = j0 + lane;
            const int o = before + __popc(starts & (0xffffffffu >> (31 - lane)));
            before += __popc(starts);
            if (j < wtot) {
                const uint4 a = list[o][0], b = list[o][1];
                const uint32_t k = j - b.x, rw = b.y & 0xffff;
                // k / rw: the quotient's distance from the next whole number is at least 0.5 / rw,
                // more than its rounding errors below 2^21
                uint32_t ky = (uint32_t)__fdividef((float)k + 0.5f, (float)rw);
                if (k >= 1u << 21) ky = k / rw;
                const uint32_t kx = k - ky * rw, st = b.z + ky * (b.y >> 16) + kx, out = base + a.w + k;
                okeys[out] = st;
                ovals[out] = a.z;
                put_mask(omask, out, tile_mask_rect<M>(a.x, a.y, (int)((b.w & 0xffff) + kx), (int)((b.w >> 16) + ky), S, s_spread));
                count(st);
            }
        }
        // the items of several rectangles: small ones by their threads, the others one at a time
        bool by_warp = cnt > 0 && xr == 0 && fits;
        if (by_warp) {
            uint32_t out = base + pre;
            const uint32_t end = out + cnt;
            by_warp = !thread_supers(cam, inv_s, ranges[item], [&](int sx, int sy, const int *rg) {
                if (out < end) {
                    const uint32_t st = (uint32_t)(cam.stile_base + sy * cam.stiles_x + sx);
                    okeys[out] = st;
                    ovals[out] = item;
                    put_mask(omask, out, tile_mask_sets(super_cols(cam, rg, sx, S), super_rows(cam, rg, sy, S), s_spread));
                    count(st);
                    ++out;
                }
            });
        }
        for (uint32_t many = __ballot_sync(0xffffffffu, by_warp); many; many &= many - 1) {
            const int o = __ffs(many) - 1;
            const uint32_t it = __shfl_sync(0xffffffffu, item, o), cn = __shfl_sync(0xffffffffu, cnt, o);
            const DevCam &c = cams[__shfl_sync(0xffffffffu, ci, o)];
            const uint32_t out = base + __shfl_sync(0xffffffffu, pre, o);
            int rg[8];
            unpack_ranges(ranges[it], rg);
            const int2 xs = super_span(rg[0], rg[1], rg[2], rg[3], inv_s), ys = super_span(rg[4], rg[5], rg[6], rg[7], inv_s);
            uint2 *sets = s_sets[threadIdx.x >> 5];
            uint32_t done = 0;
            for (int x0 = xs.x; x0 < xs.y; x0 += 32)
                for (int y0 = ys.x; y0 < ys.y; y0 += 32) {
                    __syncwarp();
                    sets[lane] = make_uint2(super_cols(c, rg, x0 + lane, S), super_rows(c, rg, y0 + lane, S));
                    __syncwarp();
                    // a lane per super-tile, row by row; 32 further is `down` rows and `right` columns
                    const int w = min(32, xs.y - x0), h = min(32, ys.y - y0), down = 32 / w, right = 32 - down * w;
                    int cy = lane / w, cx = lane - cy * w;
                    for (int k = w * h; k > 0; k -= 32) {
                        M m = 0;
                        if (lane < k) m = tile_mask_sets(sets[cx].x, sets[cy].y, s_spread);
                        const uint32_t kept = __ballot_sync(0xffffffffu, m != 0);
                        const uint32_t q = done + (uint32_t)__popc(kept & ((1u << lane) - 1u));
                        if (m != 0 && q < cn) {
                            const uint32_t st = (uint32_t)(c.stile_base + (y0 + cy) * c.stiles_x + x0 + cx);
                            okeys[out + q] = st;
                            ovals[out + q] = it;
                            put_mask(omask, out + q, m);
                            count(st);
                        }
                        done += (uint32_t)__popc(kept);
                        cx += right;
                        cy += down;
                        if (cx >= w) {
                            cx -= w;
                            ++cy;
                        }
                    }
                }
        }
    }
    __syncthreads();
    if (smem)
        for (int k = threadIdx.x; k < nst; k += kPrepThreads)
            if (sh[k]) atomicAdd(&scount[k], sh[k]);
}

// Warp-aggregated bucket atomic: the lanes with ok hold bucket bk; one atomic
// per distinct bucket of the warp adds the lanes' count to hist[bk]. Returns the
// lane's slot (old value + its rank among the lanes of its bucket). All lanes of
// the warp must call it.
__device__ __forceinline__ uint32_t bucket_add(uint32_t *hist, bool ok, int bk) {
    const unsigned peers = __match_any_sync(0xffffffffu, ok ? bk : -1);
    const int leader = __ffs(peers) - 1, lane = threadIdx.x & 31;
    uint32_t base = 0;
    if (ok && lane == leader) base = atomicAdd(&hist[bk], (uint32_t)__popc(peers));
    base = __shfl_sync(0xffffffffu, base, leader);
    return base + (uint32_t)__popc(peers & ((1u << lane) - 1u));
}

// Exclusive scan of the kOrderBuckets bucket sizes in place (warp 0; the block
// synchronises before and after).
__device__ __forceinline__ void bucket_scan(uint32_t *hist) {
    if (threadIdx.x >= 32) return;
    constexpr int kPer = (kOrderBuckets + 31) / 32;
    const int lane = threadIdx.x, b0 = lane * kPer;
    uint32_t v[kPer], sum = 0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        v[k] = b0 + k < kOrderBuckets ? hist[b0 + k] : 0u;
        sum += v[k];
    }
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    uint32_t run = incl - sum;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        if (b0 + k < kOrderBuckets) hist[b0 + k] = run;
        run += v[k];
    }
}

// Exclusive scan over [0, m) of counts held as contiguous per-thread chunks by a
// 1024-thread block: returns the prefix of the thread's chunk (s = the chunk's sum).
__device__ __forceinline__ uint32_t block_chunk_prefix(uint32_t s, uint32_t *warp_tot) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    uint32_t v = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
    }
    if (lane == 31) warp_tot[warp] = v;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = warp_tot[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        warp_tot[lane] = w;
    }
    __syncthreads();
    const uint32_t pre = v - s + (warp > 0 ? warp_tot[warp - 1] : 0u);
    __syncthreads();
    return pre;
}

// The super-tile of tile i, or -1 for a tile that a slot layout leaves unused. c: the camera
// to start looking at (0, then as the call before left it if i has not decreased).
__device__ __forceinline__ int tile_super(const DevCam *__restrict__ cams, int ncams, uint32_t inv_s, int i, int &c) {
    while (c + 1 < ncams && cams[c + 1].tile_base <= i) ++c;
    const DevCam &cm = cams[c];
    const int lt = i - cm.tile_base;
    if (lt < 0 || lt >= cm.tiles_x * cm.tiles_y) return -1;
    const int cy = lt / cm.tiles_x, cx = lt - cy * cm.tiles_x;
    return cm.stile_base + super_of(cy, inv_s) * cm.stiles_x + super_of(cx, inv_s);
}

// IdentifyFrustumRanges at super-tile granularity, block 0: each super-tile's
// [start, end) in the sorted super-tile pairs (exclusive scan of its pair count),
// and the places of the buckets in the order in which the render blocks take the
// tiles: by descending length of their super-tile's list (bucketed), so that the
// costliest tiles start first and the grid does not end on a tail of heavy tiles.
// (Measured on the 1M-Gaussian fisheye workload: 0.344 ms forward against 0.358 -
// 0.409 ms with the length capped at 16K - 1K entries and 0.424 ms in tile order.)
// A super-tile adds its tiles to its bucket; k_masks_order then places them. Blocks 1 to
// order_blocks - 1 count, per bucket, the tiles that the blocks of that kernel but the
// last will place; the others reset the fused render's unit queue. (One block that also
// walked all the tiles and the queue took 100 us on four 1920 x 1536 cameras.)
constexpr int kQueueBlock = 8 * 1024;  // queue words reset by a block
__global__ void __launch_bounds__(1024) k_tile_offsets(const DevCam *__restrict__ cams, int ncams, int S, int ntiles,
                                                       uint2 *__restrict__ srange, int nst,
                                                       uint32_t *__restrict__ misc, uint32_t *__restrict__ counts,
                                                       int order_blocks,
                                                       uint32_t *__restrict__ queue, uint32_t queue_n) {
    grid_dep_sync();
    const int t = threadIdx.x;
    __shared__ uint32_t warp_tot[32];
    __shared__ uint32_t hist[kOrderBuckets];
    // the fused render's unit queue and its counters start afresh with every binning
    if ((int)blockIdx.x >= order_blocks) {
        const uint32_t q0 = (blockIdx.x - order_blocks) * (uint32_t)kQueueBlock, q1 = min(queue_n, q0 + kQueueBlock);
        for (uint32_t i = q0 + t; i < q1; i += 1024) queue[i] = 0xffffffffu;
        return;
    }
    if (blockIdx.x == 0 && queue && t < 4) misc[kMiscFwdNext + t] = 0u;
    if (misc[kMiscStatus] & kStatusCapacity) return;
    for (int i = t; i < kOrderBuckets; i += 1024) hist[i] = 0u;
    if (blockIdx.x > 0) {
        // the tiles of k_masks_order's block blockIdx.x - 1 per bucket
        __syncthreads();
        const int i = t * order_blocks + (int)blockIdx.x - 1;
        int c = 0;
        const int st = i < ntiles ? tile_super(cams, ncams, super_inverse(S), i, c) : -1;
        bucket_add(hist, i < ntiles,
                   st >= 0 ? order_bucket(reinterpret_cast<const uint32_t *>(srange + nst)[st]) : kOrderBuckets - 1);
        __syncthreads();
        for (int b = t; b < kOrderBuckets; b += 1024) counts[(blockIdx.x - 1) * kOrderBuckets + b] = hist[b];
        return;
    }
    // super-tile ranges
    const uint32_t *scount = reinterpret_cast<const uint32_t *>(srange + nst);
    const int schunk = (nst + 1023) / 1024;
    const int sb = t * schunk, se = min(nst, sb + schunk);
    uint32_t ss = 0;
    for (int i = sb; i < se; ++i) ss += scount[i];
    uint32_t srun = block_chunk_prefix(ss, warp_tot);
    int c = 0;
    for (int i = sb; i < se; ++i) {
        const uint32_t cnt = scount[i];
        srange[i] = make_uint2(srun, srun + cnt);
        srun += cnt;
        while (c + 1 < ncams && cams[c + 1].stile_base <= i) ++c;
        const DevCam &cm = cams[c];
        const int l = i - cm.stile_base, sy = cm.stiles_x > 0 ? l / cm.stiles_x : 0, sx = l - sy * cm.stiles_x;
        const int w = min(S, cm.tiles_x - sx * S), h = min(S, cm.tiles_y - sy * S);
        if (cnt > 0 && w > 0 && h > 0) atomicAdd(&hist[order_bucket(cnt)], (uint32_t)(w * h));
    }
    __syncthreads();
    // (the last bucket's own size, the tiles without entries, is not needed)
    bucket_scan(hist);
    __syncthreads();
    for (int i = t; i < kOrderBuckets; i += 1024) misc[kMiscCount + i] = hist[i];
}

// After the sort of the super-tile pairs. Blocks [0, order_blocks) place 1024 tiles each
// in the render order: block k the tiles k, k + order_blocks, k + 2 order_blocks, ...,
// in each bucket behind those of the blocks before it (counts), so that tiles rendered at
// the same time lie apart in the image. The order is part of a gradient's rounding: the
// sums of a Gaussian over hundreds of tiles are added as the tiles finish. With runs of
// neighbouring tiles in turn, placed as their blocks came, the scale gradients of needles
// near the cameras, small differences of large sums, moved: four 1920 x 1536 cameras, 6M
// Gaussians, the means of four runs by 1.4e-6 of the gradients' norm and single ones by
// 4e-3 of their size, where the runs of one order give 0.7e-6 and 1e-3. (The same time.)
// The others: the or of every 32 sorted pairs' tile masks (a warp per group): the
// render's list scan skips the groups without an entry of its tile.
__global__ void __launch_bounds__(256) k_masks_order(const DevCam *__restrict__ cams, int ncams, int S, int ntiles,
                                                     const uint2 *__restrict__ srange, uint32_t *__restrict__ order,
                                                     int order_blocks, const uint32_t *__restrict__ counts,
                                                     const uint32_t *__restrict__ mask, int words,
                                                     const uint32_t *__restrict__ misc, uint32_t *__restrict__ any) {
    grid_dep_sync();
    if (misc[kMiscStatus] & kStatusCapacity) return;
    const int t = threadIdx.x, lane = t & 31;
    if ((int)blockIdx.x < order_blocks) {
        __shared__ uint32_t hist[kOrderBuckets];
        const uint32_t inv_s = super_inverse(S);
        const int i0 = t * order_blocks + (int)blockIdx.x;
        int c = 0;
        uint2 r[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * 256 * order_blocks, st = i < ntiles ? tile_super(cams, ncams, inv_s, i, c) : -1;
            r[u] = st >= 0 ? srange[st] : make_uint2(0u, 0u);
        }
        if (t < kOrderBuckets) {
            uint32_t at = misc[kMiscCount + t];
#pragma unroll 8
            for (int k = 0; k < (int)blockIdx.x; ++k) at += counts[k * kOrderBuckets + t];
            hist[t] = at;
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * 256 * order_blocks;
            const uint32_t at = bucket_add(hist, i < ntiles, order_bucket(r[u].y - r[u].x));
            if (i < ntiles) order[at] = (uint32_t)i;
        }
        return;
    }
    // a warp takes four groups at a time, their loads in flight together
    constexpr int G = 4;
    const uint64_t n = misc[kMiscPairs], step = (uint64_t)(gridDim.x - order_blocks) * (256u * G);
    for (uint64_t i0 = ((uint64_t)(blockIdx.x - order_blocks) * 8u + (t >> 5)) * (32u * G); i0 < n; i0 += step) {
        uint32_t m[G][2];
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const uint64_t i = i0 + 32 * g + lane;
            m[g][0] = m[g][1] = 0u;
            if (i < n) {
                if (words == 1) {
                    m[g][0] = mask[i];
                } else {
                    const uint2 v = reinterpret_cast<const uint2 *>(mask)[i];
                    m[g][0] = v.x;
                    m[g][1] = v.y;
                }
            }
        }
#pragma unroll
        for (int g = 0; g < G; ++g)
            for (int w = 0; w < words; ++w) {
                const uint32_t v = __reduce_or_sync(0xffffffffu, w ? m[g][1] : m[g][0]);
                if (lane == 0 && i0 + 32 * g < n) any[(i0 / 32 + g) * words + w] = v;
            }
    }
}

// One block: the backward's units and their schedule. A tile whose forward walk
// covered W > 0 list entries and passed the checkpoints B_1 < ... < B_m < W
// has the units k = 0..m, entries [B_k, B_{k+1}) with B_0 = 0 and B_{m+1} = W.
// The forward leaves per tile their number and schedule buckets (unit_rec: the
// bucket of each unit's cost, the (entry, warp) pairs whose hit byte it set in
// the unit: a backward warp walks those steps, so a dense tile's unit costs
// more than a sparse one's of the same length). The units are ordered by
// descending cost, units[slot] = tile << 4 | k. Also sets the unit count and
// resets the counter the persistent backward blocks take units from.
__global__ void __launch_bounds__(1024) k_bwd_order(const uint4 *__restrict__ unit_rec, int ntiles,
                                                    uint32_t *__restrict__ misc, uint32_t *__restrict__ order) {
    grid_dep_sync();
    __shared__ uint32_t hist[kOrderBuckets];
    __shared__ uint32_t s_total;
    if (misc[kMiscStatus] & kStatusCapacity) return;
    const int t = threadIdx.x;
    for (int i = t; i < kOrderBuckets; i += 1024) hist[i] = 0u;
    if (t == 0) s_total = 0u;
    __syncthreads();
    const int chunk = (ntiles + 1023) / 1024;
    const int b = t * chunk, e = min(ntiles, b + chunk);
    constexpr int G = 4;  // tiles whose records are loaded together
    for (int pass = 0; pass < 2; ++pass) {
        uint32_t mine = 0;
        for (int c0 = 0; c0 < chunk; c0 += G) {  // the same trip counts in every lane (warp-wide atomics)
            uint4 r[G];
#pragma unroll
            for (int u = 0; u < G; ++u) {
                const int i = b + c0 + u;
                r[u] = c0 + u < chunk && i < e ? unit_rec[i] : make_uint4(0u, 0u, 0u, 0u);
            }
#pragma unroll
            for (int u = 0; u < G; ++u) {
                const int i = b + c0 + u;
                const uint32_t units = min((r[u].w >> (8 * (kUnitCountByte & 3))) & 0xffu, (uint32_t)kCkptMax + 1u);
#pragma unroll
                for (int k = 0; k <= kCkptMax; ++k) {
                    if (!__any_sync(0xffffffffu, (uint32_t)k < units)) break;
                    const bool ok = (uint32_t)k < units;
                    const uint32_t word = k < 4 ? r[u].x : (k < 8 ? r[u].y : r[u].z);
                    const int bk = min((int)((word >> (8 * (k & 3))) & 0xffu), kOrderBuckets - 1);
                    const uint32_t slot = bucket_add(hist, ok, bk);
                    if (pass == 1 && ok) order[slot] = ((uint32_t)i << 4) | (uint32_t)k;
                }
                mine += units;
            }
        }
        if (pass == 0) {
            atomicAdd(&s_total, mine);
            __syncthreads();
            bucket_scan(hist);
        }
        __syncthreads();
    }
    if (t == 0) {
        misc[kMiscUnits] = s_total;
        misc[kMiscUnitNext] = 0u;
    }
}

}  // namespace

cudaError_t launch_preprocess(const geer_workspace *ws, const geer_gaussians *g, cudaStream_t s) {
    const int64_t nblk = prep_blocks(g->n);
    if (nblk == 0) return cudaSuccess;
    const Params prm = ws->params;
    const bool splat = prm.assoc != GEER_ASSOC_PBF || prm.alpha_model != GEER_ALPHA_EXACT;
#define GEER_PREP_LAUNCH(D)                                                                                      \
    {                                                                                                            \
        const int smem = kPrepThreads * ShRows<D>::kStride * (int)sizeof(float);                               \
        auto *kern = splat ? k_preprocess<D, true> : k_preprocess<D, false>;                                     \
        if (smem > 48 * 1024) {                                                                                  \
            const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);  \
            if (e != cudaSuccess) return e;                                                                      \
        }                                                                                                        \
        launch_k(kern, dim3((unsigned)nblk), dim3(kPrepThreads), smem, s, ws->d_cams, ws->n_cams,                 \
                 ws->d_tile_tab, prm, g->mean, g->scale, g->quat, g->opacity, g->sh, g->n, ws->d_rec,            \
                 ws->d_ranges, ws->trains ? ws->d_gacc : nullptr, ws->d_count, ws->d_key,                    \
                 ws->d_blocksum, nblk);                                                                   \
    }
    switch (g->sh_degree) {
        case 0: GEER_PREP_LAUNCH(0); break;
        case 1: GEER_PREP_LAUNCH(1); break;
        case 2: GEER_PREP_LAUNCH(2); break;
        default: GEER_PREP_LAUNCH(3); break;
    }
#undef GEER_PREP_LAUNCH
    return cudaGetLastError();
}

// Few enough items for one block or cluster to do the work of launch_bin_front, launch_depth_sort
// and launch_count_pairs (k_small_front, launched as launch_bin_front).
bool small_front(const geer_workspace *ws) { return (int64_t)ws->n_cams * ws->n_gauss <= kClusterItems; }

static cudaError_t launch_small_front(const geer_workspace *ws, cudaStream_t s) {
    const int items = (int)(ws->n_cams * ws->n_gauss);
    static_assert(kSmallThreads <= kSmallItems && kSmallItems <= 4 * kSmallThreads &&
                      kClusterItems <= 4 * kCluster * kSmallThreads && kClusterItems <= 65536,
                  "items a thread, 16-bit ids");
    const auto launch = [&](auto *kern, int k, int blocks) {
        const int smem = 2 * (int)sizeof(uint32_t) * kSmallThreads / 32 * kRadix + 6 * k * kSmallThreads;
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        launch_cluster(kern, dim3((unsigned)blocks), dim3(kSmallThreads), smem, s, (unsigned)blocks, ws->d_cams, ws->n_gauss, items, ws->super_size,
                 ws->d_count, ws->d_key, ws->d_ranges, ws->d_misc, ws->d_iid[0], ws->d_iid[1], ws->d_ikey[0],
                 ws->d_ikey[1], ws->d_blocksum2, reinterpret_cast<uint32_t *>(ws->d_srange + ws->n_stiles),
                 ws->n_stiles, ws->cap_pairs);
        return cudaGetLastError();
    };
    if (items <= kSmallThreads) return launch(k_small_front<1, 1>, 1, 1);
    if (items <= kSmallItems) return launch(k_small_front<4, 1>, 4, 1);
    if (items <= kCluster * kSmallThreads) return launch(k_small_front<1, kCluster>, 1, kCluster);
    if (items <= 2 * kCluster * kSmallThreads) return launch(k_small_front<2, kCluster>, 2, kCluster);
    return launch(k_small_front<4, kCluster>, 4, kCluster);
}

cudaError_t launch_bin_front(const geer_workspace *ws, cudaStream_t s) {
    if (small_front(ws)) return launch_small_front(ws, s);
    const int64_t nblk = prep_blocks(ws->n_gauss);
    launch_k(k_scan_blocks, dim3(1), dim3(1024), 0, s, ws->d_blocksum, nblk * ws->n_cams, ws->d_misc, ws->d_srange,
             ws->n_stiles, ws->cap_pairs, 0, nullptr, 0);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || nblk == 0) return e;
    launch_k(k_compact, dim3((unsigned)((nblk + kCompact - 1) / kCompact), (unsigned)ws->n_cams), dim3(kPrepThreads), 0, s, ws->n_gauss, ws->d_count,
             ws->d_key, ws->d_blocksum, nblk, ws->d_ikey[0], ws->d_iid[0]);
    return cudaGetLastError();
}

cudaError_t launch_count_pairs(const geer_workspace *ws, cudaStream_t s) {
    if (small_front(ws)) return cudaSuccess;
    const int64_t m = prep_blocks((int64_t)ws->n_cams * ws->n_gauss);
    if (m > 0) {
        launch_k(k_gather_counts, dim3((unsigned)((m + kGather - 1) / kGather)), dim3(kPrepThreads), 0, s, ws->d_cams,
                 ws->n_gauss, ws->super_size, ws->d_iid[0], ws->d_iid[1], ws->d_ranges, ws->d_misc, ws->d_blocksum2,
                 ws->d_blocksum3, ws->d_ikey[0], ws->d_ikey[1]);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    // super-tile pairs: emission offsets and the capacity check; tile associations: the count P
    launch_k(k_scan_blocks, dim3(2), dim3(1024), 0, s, ws->d_blocksum2, m, ws->d_misc, nullptr, 0, ws->cap_pairs, 1,
             ws->d_blocksum3, 2);
    return cudaGetLastError();
}

// The blocks that place 1024 tiles each in the render order, and their bucket counts (all
// blocks' but the last one's), which live in the scratch words behind the walk records.
static int order_blocks(const geer_workspace *ws) { return (int)((ws->n_tiles + 1023) / 1024); }
static uint32_t *order_counts(const geer_workspace *ws) {
    static_assert(kOrderBuckets < 1024, "a word per tile holds a row of counts per 1024 tiles");
    return reinterpret_cast<uint32_t *>(ws->d_tile_walk + ws->n_tiles);
}

cudaError_t launch_duplicate(const geer_workspace *ws, cudaStream_t s) {
    const int64_t m = prep_blocks((int64_t)ws->n_cams * ws->n_gauss);
    uint32_t *scount = reinterpret_cast<uint32_t *>(ws->d_srange + ws->n_stiles);
    if (m > 0) {
        const size_t smem = ws->n_stiles <= kSmemTiles ? sizeof(uint32_t) * ws->n_stiles : 0;
        auto *kern = mask_words(ws->super_size) == 1 ? k_duplicate<uint32_t> : k_duplicate<uint64_t>;
        // the counters come beside ~10 KB of lists: from ~9780 super-tiles on more than the 48 KB of a plain launch
        if (smem > 32 * 1024) {
            const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                       (int)sizeof(uint32_t) * kSmemTiles);  // (the same for every caller)
            if (e != cudaSuccess) return e;
        }
        const int64_t blocks = std::min<int64_t>(m, (int64_t)ws->num_sms * 4);
        launch_k(kern, dim3((unsigned)blocks),
                 dim3(kPrepThreads), smem, s, ws->d_cams, ws->n_gauss, ws->super_size, ws->d_iid[0], ws->d_iid[1],
                 ws->d_ikey[0], ws->d_ikey[1], ws->d_ranges, ws->d_misc, ws->d_blocksum2, ws->d_keys[0], ws->d_vals[0], ws->d_smask[0], scount,
                 (int)ws->n_stiles, ws->cap_pairs);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    const uint32_t queue_n = ws->trains ? (uint32_t)(ws->n_tiles * (kCkptMax + 1)) : 0u;
    const int first = std::max(1, order_blocks(ws));
    launch_k(k_tile_offsets, dim3(first + (queue_n + kQueueBlock - 1) / kQueueBlock), dim3(1024), 0, s, ws->d_cams,
             ws->n_cams, ws->super_size, (int)ws->n_tiles, ws->d_srange, (int)ws->n_stiles, ws->d_misc,
             order_counts(ws), first, ws->trains ? ws->d_bwd_order : nullptr, queue_n);
    return cudaGetLastError();
}

cudaError_t launch_masks_order(const geer_workspace *ws, cudaStream_t s) {
    const int64_t blocks = std::min<int64_t>(std::max<int64_t>(1, (ws->cap_pairs + 255) / 256), (int64_t)ws->num_sms * 8);
    launch_k(k_masks_order, dim3((unsigned)(blocks + order_blocks(ws))), dim3(256), 0, s, ws->d_cams, ws->n_cams,
             ws->super_size, (int)ws->n_tiles, ws->d_srange, ws->d_tile_order, order_blocks(ws),
             (const uint32_t *)order_counts(ws), (const uint32_t *)ws->d_smask[ws->sorted_buf], mask_words(ws->super_size), ws->d_misc, ws->d_sany);
    return cudaGetLastError();
}

cudaError_t launch_bwd_order(const geer_workspace *ws, cudaStream_t s) {
    if (ws->n_tiles == 0) return cudaSuccess;
    launch_k(k_bwd_order, dim3(1), dim3(1024), 0, s, ws->d_unit_rec, (int)ws->n_tiles, ws->d_misc,
             ws->d_bwd_order);
    return cudaGetLastError();
}

}  // namespace geer
