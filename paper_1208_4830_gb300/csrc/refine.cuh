// refine.cuh -- FP64 images and magnification from FP32 roots.
//
// What bounds FP64 work here: the FP64 pipe takes one warp instruction per 64 cycles from a warp (19
// cycles per SM over all its warps) whatever the number of active lanes, and a divergent warp pays
// for the union of its lanes' paths. So FP64 operations are spent only where their digits reach the
// result, the lens equation at the images, and an epoch's five roots are spread over five lanes.
//
// refine_root takes one root known to FP32 accuracy to FP64: Newton steps on the lens equation whose
// residual is FP64 and whose Jacobian and correction are FP32 (iterative refinement: each step
// shrinks the error by the FP32 Jacobian's relative error, about 2e-7 / |det J|, and quadratically)
// until the correction is below kRefineStep min(1, |det J|) of the distance to the nearer lens; the
// Jacobian at the last point in FP64, advanced by that last correction to first order, gives det J.
// 16 FP64 instructions for the first step, 20 for each further one and about 20 for the last one's Jacobian,
// against some 250 per root and sweep of a root iteration in FP64. FP64 chi^2 of 4096 x 2000: 68.6 ms with the
// quintic solved in FP64, 8.4 ms so; one event's curve of 400 epochs: 1129 us, 189 us.
#pragma once

#include "forward.cuh"

namespace sblm {

constexpr float kRefineStep = 1e-9f;

// Lenses and sources whose epochs are refined; others (and sources within 1e-6 of a lens, where the
// quintic's leading coefficient vanishes) take the general FP64 solver. The range is the one over
// which refined magnifications were compared with that solver and with 40-digit arithmetic, 20M
// epochs of caustic-crossing trajectories: beyond it (q below 5e-5 above all) the general solver's
// own roots are uncertain and its results are what is to be returned.
constexpr float kRefineQLo = 5e-5f, kRefineQHi = 30.f, kRefineDLo = 0.25f, kRefineDHi = 10.f, kRefineZeta = 64.f;

__device__ __forceinline__ bool refine_lens(float d, float q) {
    return q >= kRefineQLo && q <= kRefineQHi && d >= kRefineDLo && d <= kRefineDHi;
}
__device__ __forceinline__ bool refine_source(cx<float> zeta, float d) {
    return norm2(zeta) <= kRefineZeta * kRefineZeta && norm2(zeta) >= 1e-12f &&
           norm2(mk<float>(zeta.re - d, zeta.im)) >= 1e-12f;
}

// one root in FP64: its position from the primary (z) and from the secondary (w = z - d), both
// advanced by every correction so that the one that is small keeps its relative precision
struct Refined {
    cx<double> z, w;
    double det;  // det J at the root
    bool image;  // the corrections converged: a solution of the lens equation
};

// One Newton step on the lens equation at (z, w), r1 and r2 the reciprocals of norm2(z) and norm2(w): the FP64
// residual's correction by the FP32 Jacobian, and the FP32 terms it was taken from
struct LensStep {
    cx<float> delta, u, v, K;
    float dj_abs, dj_rcp;
};
__device__ __forceinline__ LensStep lens_step(cx<double> z, cx<double> w, double r1, double r2, cx<double> zeta, double q) {
    LensStep o;
    const double qr2 = q * r2;
    // u = 1/conj(z) = z r1, v = 1/(d - conj(z)) = -w r2; f = z - u + q v - zeta
    cx<double> f;
    f.re = fma(-w.re, qr2, fma(-z.re, r1, z.re)) - zeta.re;
    f.im = fma(-w.im, qr2, fma(-z.im, r1, z.im)) - zeta.im;
    const float qf = (float)q, r1f = (float)r1, r2f = (float)r2;
    const cx<float> zf = mk<float>((float)z.re, (float)z.im), wf = mk<float>((float)w.re, (float)w.im);
    const cx<float> ff = mk<float>((float)f.re, (float)f.im);
    o.u = r1f * zf;
    o.v = (-r2f) * wf;
    o.K = o.u * o.u + qf * (o.v * o.v);
    const float dj = 1.f - norm2(o.K);
    o.dj_abs = fabs(dj);
    const cx<float> num = o.K * conj(ff) - ff;
    o.dj_rcp = rcp(o.dj_abs);
    o.delta = (dj < 0.f ? -o.dj_rcp : o.dj_rcp) * num;
    return o;
}

// Newton steps on the lens equation from (z, w); at most `cap` corrections. SHORT_FIRST: the residual of the
// first correction to 2^-40 only, enough for an error of FP32's size at an image with |det J| above 0.1 (below 0.03
// it would cost a third correction).
template <bool SHORT_FIRST>
__device__ __forceinline__ Refined refine_root(cx<double> z, cx<double> w, cx<double> zeta, double q, int cap) {
    Refined o;
    o.image = false;
    o.det = 1.0;
    if (SHORT_FIRST) {
        const cx<float> delta = lens_step(z, w, rcp_start(norm2(z)), rcp_start(norm2(w)), zeta, q).delta;
        z = mk<double>(z.re + (double)delta.re, z.im + (double)delta.im);
        w = mk<double>(w.re + (double)delta.re, w.im + (double)delta.im);
        --cap;
    }
    const float qf = (float)q;
    const float zeta_abs = sqrt_(norm2(mk<float>((float)zeta.re, (float)zeta.im)));
#pragma unroll 1
    for (int it = 0;; ++it) {
        const double n1 = norm2(z), n2 = norm2(w);
        const double r1 = rcp_normal(n1), r2 = rcp_normal(n2);
        const LensStep s = lens_step(z, w, r1, r2, zeta, q);
        const float d2 = norm2(s.delta);
        if (!isfinite(d2)) break;
        // stop at the step bound, or at the rounding level of f's FP64 evaluation
        const float n1f = (float)n1, n2f = (float)n2;
        const float scale = sqrt_(n1f) + sqrt_((float)r1) + qf * sqrt_((float)r2) + zeta_abs;
        const float lim =
            fmax(kRefineStep * fmin(s.dj_abs, 1.f) * sqrt_(fmin(n1f, n2f)), 1e-15f * scale * s.dj_rcp);
        const bool last = d2 <= lim * lim;
        if (last) {
            // K in FP64 at (z, w), and det J advanced by delta: dK = 2 conj(delta) (q v^3 - u^3)
            const double uu = r1 * r1, vv = q * r2 * r2;
            const double kr = fma(fma(z.re, z.re, -(z.im * z.im)), uu, fma(w.re, w.re, -(w.im * w.im)) * vv);
            const double ki = fma(z.re * z.im, uu, (w.re * w.im) * vv);
            const cx<float> dK = (2.f * conj(s.delta)) * (qf * (s.v * s.v * s.v) - s.u * s.u * s.u);
            const float ddet = -2.f * (s.K.re * dK.re + s.K.im * dK.im);
            o.det = fma(-4.0 * ki, ki, fma(-kr, kr, 1.0)) + (double)ddet;
            o.image = true;
        }
        if (!last && it >= cap) break;
        const double dr = (double)s.delta.re, di = (double)s.delta.im;
        z = mk<double>(z.re + dr, z.im + di);
        w = mk<double>(w.re + dr, w.im + di);
        if (last) break;
    }
    o.z = z;
    o.w = w;
    return o;
}

// (z, w = z - d) in FP64 of a root found in FP32 with the separation df = (float)d: next to the
// secondary the offset z - df is the accurate part
__device__ __forceinline__ void start_from_fp32(cx<float> zf, double d, cx<double>& z, cx<double>& w) {
    const float df = (float)d;
    const bool near2 = fabs(zf.re) > fabs(zf.re - df);
    w = mk<double>((double)zf.re - (near2 ? (double)df : d), (double)zf.im);
    z = mk<double>(near2 ? d + w.re : (double)zf.re, (double)zf.im);
}

// FP64 magnification of an epoch whose images FP32 identified without a trigger: the images in the
// bit mask `images` of the FP32 roots rp refined one after the other. False when a root does not
// converge next to where FP32 had it (within 1e-3 of the distance to its nearest neighbour) or the
// parities do not sum to -1: the epoch then goes to the re-solve.
__device__ __forceinline__ bool refine_images(const Root<float> rp[5], unsigned images, cx<double> zeta, double d,
                                              double q, double* A) {
    double sum = 0.0;
    int parity = 0;
    bool ok = true;
#pragma unroll 1
    while (images) {  // the set bits only: 3 images in different slots of a warp's lanes take 3 passes
        const int i = __ffs(images) - 1;
        images &= images - 1;
        Root<float> r = rp[0];
#pragma unroll
        for (int k = 1; k < 5; ++k)
            if (i == k) r = rp[k];
        float gap2 = INFINITY;
#pragma unroll
        for (int k = 0; k < 5; ++k) gap2 = k == i ? gap2 : fmin(gap2, norm2(root_diff(rp[k], r)));
        cx<double> z, w;
        w = mk<double>(r.local ? (double)r.w.re : (double)r.z.re - d, r.local ? (double)r.w.im : (double)r.z.im);
        z = mk<double>(r.local ? d + w.re : (double)r.z.re, r.local ? w.im : (double)r.z.im);
        const Refined f = refine_root<true>(z, w, zeta, q, 4);
        const cx<float> moved = mk<float>((float)(f.w.re - w.re), (float)(f.w.im - w.im));
        ok = ok && f.image && norm2(moved) <= 1e-6f * gap2;
        const double a = fabs(f.det);
        sum += rcp_normal(a);
        parity += f.det < 0.0 ? -1 : 1;
    }
    *A = sum;
    return ok && parity == -1;
}

// ------------------------------------------------------------------------------------------
// The re-solve of queued epochs: one warp takes six, five lanes each (lanes 30 and 31 idle), a lane
// per root. Every lane of the warp calls it.
// ------------------------------------------------------------------------------------------
constexpr int kResolveLanes = 5, kResolvePerWarp = 6;
// an epoch whose roots the quintic's FP64 rounding noise blurs by more than this share of the
// smallest gap between them goes to the general solver (0.02% of the re-solved epochs of the sweep)
constexpr float kTightRoots = 3e-3f;
// an epoch with an image at |det J| below this goes to the general solver: A's rounding error there,
// about 2^-53 / (det J)^2 relative, reaches 1e-9, and which way it falls is that solver's (0.03% of the
// re-solved epochs; at 1e-3 four times as many, each of which holds up a small call by 100 us)
constexpr float kFoldDet = 5e-4f;
// least relative lens-equation residual at which a root of the quintic counts as spurious: computed
// in FP32 after the images were divided out, and in FP64 after the FP64 root iteration
constexpr float kSpuriousResidual32 = 1e-4f;
constexpr double kSpuriousResidual64 = 1e-6;

__device__ __forceinline__ cx<float> shfl(cx<float> a, int src) {
    return mk<float>(__shfl_sync(0xffffffffu, a.re, src), __shfl_sync(0xffffffffu, a.im, src));
}
__device__ __forceinline__ cx<double> shfl(cx<double> a, int src) {
    return mk<double>(__shfl_sync(0xffffffffu, a.re, src), __shfl_sync(0xffffffffu, a.im, src));
}

// Clear `image` on a lane whose solution a lower lane of the group found too (coinciding to 3e-6 of
// the distances to both lenses). Returns whether any lane of the warp dropped one, by lane bit.
__device__ __forceinline__ unsigned drop_duplicates(Refined& f, int base, int r) {
    const cx<float> zf = mk<float>((float)f.z.re, (float)f.z.im), wf = mk<float>((float)f.w.re, (float)f.w.im);
    bool dup = false;
#pragma unroll
    for (int s = 1; s < 5; ++s) {
        const int j = r + s < 5 ? r + s : r + s - 5;
        const cx<float> zo = shfl(zf, base + j), wo = shfl(wf, base + j);
        const bool io = __shfl_sync(0xffffffffu, (int)f.image, base + j) != 0;
        dup = dup || (io && f.image && j < r && norm2(zo - zf) <= 1e-11f * fmin(norm2(zo), norm2(zf)) &&
                      norm2(wo - wf) <= 1e-11f * fmin(norm2(wo), norm2(wf)));
    }
    if (dup) f.image = false;
    return __ballot_sync(0xffffffffu, dup);
}

// images of a group and the sum of their parities
__device__ __forceinline__ void count_images(const Refined& f, int base, int* count, int* parity) {
    const unsigned all = __ballot_sync(0xffffffffu, f.image) >> base & 31u;
    const unsigned neg = __ballot_sync(0xffffffffu, f.image && f.det < 0.0) >> base & 31u;
    *count = __popc(all);
    *parity = __popc(all) - 2 * __popc(neg);
}

// sum over the group's images of 1/|det J|, in root order, in every lane of the group
__device__ __forceinline__ double image_sum(const Refined& f, int base) {
    const double a = f.image ? rcp_normal(fabs(f.det)) : 0.0;
    double sum = 0.0;
#pragma unroll
    for (int s = 0; s < 5; ++s) sum += __shfl_sync(0xffffffffu, a, base + s);
    return sum;
}

// The two roots of the quintic that remain once three images (sum `zs`, product `zp`) are divided out,
// from its coefficients; `which` selects one: whether that root is far from solving the lens equation.
__device__ __forceinline__ bool remaining_root_spurious(cx<double> zs, cx<double> zp, cx<double> zeta, double d,
                                                        double q, int which) {
    const cx<double> s = conj(zeta);
    const double m = 1.0 + q;
    const cx<double> n1 = mk<double>(fma(-d, s.re, m), -d * s.im), k2 = mk<double>(s.re - d, s.im);
    const cx<double> k1 = mk<double>(fma(d, d, n1.re), n1.im);
    const cx<double> c5 = s * k2;
    const cx<double> c4 = s * k1 + n1 * k2 - zeta * c5 - k2 - q * s;
    const double rc = rcp_normal(norm2(c5));
    const cx<double> ic5 = mk<double>(c5.re * rc, -c5.im * rc);
    const cx<double> h = -0.5 * (c4 * ic5 + zs);
    const cx<double> den = c5 * zp;  // the quintic's roots multiply to d^2 zeta / c5
    const double rd = rcp_normal(norm2(den)) * (d * d);
    const cx<double> P = zeta * mk<double>(den.re * rd, -den.im * rd);
    const cx<double> D = h * h - P;
    // the square root in FP32: the two roots to FP32 accuracy relative to their distance
    const cx<float> Df = mk<float>((float)D.re, (float)D.im);
    const float mod = sqrt_(norm2(Df));
    float sr = sqrt_(fmax(0.5f * (mod + Df.re), 0.f)), si = sqrt_(fmax(0.5f * (mod - Df.re), 0.f));
    if (Df.im < 0.f) si = -si;
    if (which & 1) {
        sr = -sr;
        si = -si;
    }
    Root<float> t;
    t.local = true;
    t.z = mk<float>((float)h.re + sr, (float)h.im + si);
    t.w = mk<float>((float)(h.re - d) + sr, (float)h.im + si);
    cx<float> ff, K;
    float qt;
    const cx<float> zf = mk<float>((float)zeta.re, (float)zeta.im);
    lens_terms(t, zf, (float)d, (float)q, ff, K, qt);
    const float az2 = norm2(t.z);
    const float scale = sqrt_(az2) + rsqrt_(az2) + qt + sqrt_(norm2(zf));
    return norm2(ff) > kSpuriousResidual32 * kSpuriousResidual32 * scale * scale;  // NaN: not known to be
}

// Aberth-Ehrlich iteration in FP64 over the group's lanes (every root corrected at once from the
// previous positions of the others) of the lanes with `move`, from z; the others only repel
static __device__ __noinline__ cx<double> lane_aberth(cx<double> z, bool move, cx<double> zeta, double d, double q, int base,
                                               int r) {
    cx<double> c[6];
    quintic_coefficients(zeta, d, 1.0, q, c);
    double ac[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) ac[k] = sqrt_(norm2(c[k]));
#pragma unroll 1
    for (int it = 0; it < 12; ++it) {
        if (!__any_sync(0xffffffffu, move)) break;
        cx<double> S = mk<double>(0.0, 0.0);
#pragma unroll
        for (int s = 1; s < 5; ++s) S = S + inv(z - shfl(z, base + (r + s < 5 ? r + s : r + s - 5)));
        if (!move) continue;
        cx<double> p, dp;
        horner2(c, z, p, dp);
        const double az = sqrt_(norm2(z));
        double eb = ac[5];
#pragma unroll
        for (int k = 4; k >= 0; --k) eb = eb * az + ac[k];
        const double lim = (double)kNoise * Eps<double>::value * eb;
        if (norm2(p) <= lim * lim) {
            move = false;
            continue;
        }
        const cx<double> ratio = div(p, dp);
        cx<double> dz = div(ratio, mk<double>(1.0, 0.0) - ratio * S);
        if (!finite2(dz)) dz = finite2(ratio) ? ratio : mk<double>(0.0, 0.0);
        z = z - dz;
        move = !(norm2(dz) <= 1e-24 * norm2(z));
    }
    return z;
}

// Magnification of the epoch of a group of five lanes (lane `base` + r holds the FP32 root zf; all
// lanes the lens (d, q) and source zeta), in every lane of the group. First every root is refined:
// five different solutions of the lens equation are all there are; three with the right parities are
// complete when the quintic's other two roots do not solve it. What this leaves open (0.5% of the
// re-solved epochs) is decided from FP64 roots of the quintic. Returns false where that is open too
// (or the lens lies outside the range): the general solver's. Results do not depend on what the
// other groups of the warp hold.
__device__ __forceinline__ bool resolve_group(cx<float> zf, bool valid, cx<double> zeta, double d, double q, double* A) {
    const int lane = threadIdx.x & 31;
    const int grp = lane / kResolveLanes, base = grp * kResolveLanes, r = lane - base;
    const cx<float> zetaf = mk<float>((float)zeta.re, (float)zeta.im);
    const bool in_range = valid && refine_lens((float)d, (float)q) && refine_source(zetaf, (float)d);
    if (!__any_sync(0xffffffffu, in_range)) return false;
    // the smallest gap between this root and the others, and the quintic's rounding noise at it,
    // kNoise eps prod (|z| + |z_j|) / prod |z - z_j| (j = i included above)
    const float az = sqrt_(norm2(zf));
    float num = 2.f * az, den = 1.f, gap = INFINITY;
#pragma unroll
    for (int s = 1; s < 5; ++s) {
        const cx<float> o = shfl(zf, base + (r + s < 5 ? r + s : r + s - 5));
        const float dd = sqrt_(norm2(zf - o));
        num *= az + sqrt_(norm2(o));
        den *= dd;
        gap = fmin(gap, dd);
    }
    const bool loose = (kNoise * 1.1102230e-16f) * num <= kTightRoots * den * gap;  // false for NaN
    const unsigned loose_lanes = __ballot_sync(0xffffffffu, loose) >> base & 31u;
    const bool open = in_range && loose_lanes == 31u;
    if (!__any_sync(0xffffffffu, open)) return false;
    cx<double> z, w;
    start_from_fp32(zf, d, z, w);
    Refined f;
    f.image = false;
    f.z = z;
    f.w = w;
    f.det = 1.0;
    if (open) f = refine_root<false>(z, w, zeta, q, 8);
    drop_duplicates(f, base, r);
    int count, parity;
    count_images(f, base, &count, &parity);
    bool done = open && count == 5 && parity == -1;
    const bool three = open && count == 3 && parity == -1;
    if (__any_sync(0xffffffffu, three)) {
        cx<double> zs = mk<double>(0.0, 0.0), zp = mk<double>(1.0, 0.0);
        const cx<double> mine_s = f.image ? f.z : zs, mine_p = f.image ? f.z : zp;
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            zs = zs + shfl(mine_s, base + j);
            zp = zp * shfl(mine_p, base + j);
        }
        const bool sp = remaining_root_spurious(zs, zp, zeta, d, q, r);
        const unsigned b = __ballot_sync(0xffffffffu, sp) >> base & 3u;
        done = done || (three && b == 3u);
    }
    double sum = image_sum(f, base);
    bool fold = (__ballot_sync(0xffffffffu, f.image && fabs((float)f.det) < kFoldDet) >> base & 31u) != 0;
    if (__any_sync(0xffffffffu, open && !done && !fold)) {
        const bool mine = open && !done && !fold;
        const cx<double> x = lane_aberth(f.image ? f.z : z, mine && !f.image, zeta, d, q, base, r);
        float gap2 = INFINITY;
#pragma unroll
        for (int s = 1; s < 5; ++s) {
            const cx<double> o = x - shfl(x, base + (r + s < 5 ? r + s : r + s - 5));
            gap2 = fmin(gap2, norm2(mk<float>((float)o.re, (float)o.im)));
        }
        const cx<double> xw = mk<double>(x.re - d, x.im);
        Refined h;
        h.image = false;
        h.z = x;
        h.w = xw;
        h.det = 1.0;
        if (mine) h = refine_root<false>(x, xw, zeta, q, 6);
        const cx<float> moved = mk<float>((float)(h.w.re - xw.re), (float)(h.w.im - xw.im));
        h.image = h.image && norm2(moved) <= 0.25f * gap2;
        const unsigned dups = drop_duplicates(h, base, r) >> base & 31u;
        bool sp = true;
        if (!h.image) {
            Root<double> t;
            t.local = false;
            t.z = x;
            t.w = xw;
            cx<double> ff, K;
            double qt;
            lens_terms(t, zeta, d, q, ff, K, qt);
            const double az2 = norm2(x);
            const double scale = sqrt_(az2) + rsqrt_(az2) + qt + sqrt_(norm2(zeta));
            sp = norm2(ff) > kSpuriousResidual64 * kSpuriousResidual64 * scale * scale;
        }
        const bool all_sp = (__ballot_sync(0xffffffffu, sp) >> base & 31u) == 31u;
        count_images(h, base, &count, &parity);
        const double sum2 = image_sum(h, base);
        if (mine && dups == 0 && parity == -1 && (count == 5 || (count == 3 && all_sp))) {
            sum = sum2;
            done = true;
        }
        if (mine) fold = false;
        const unsigned b = __ballot_sync(0xffffffffu, mine && h.image && fabs((float)h.det) < kFoldDet) >> base & 31u;
        fold = fold || b != 0;
    }
    *A = sum;
    return done && !fold;
}

// resolve_group's first stage by one thread, its roots one after the other: for callers that re-solve a
// few epochs each in its own thread. False where it is open: the general solver's.
__device__ __forceinline__ bool resolve_thread(const cx<float>* z32, cx<double> zeta, double d, double q, double* A) {
    const cx<float> zetaf = mk<float>((float)zeta.re, (float)zeta.im);
    if (!refine_lens((float)d, (float)q) || !refine_source(zetaf, (float)d)) return false;
    for (int i = 0; i < 5; ++i) {
        const float az = sqrt_(norm2(z32[i]));
        float num = 2.f * az, den = 1.f, gap = INFINITY;
        for (int j = 0; j < 5; ++j) {
            if (j == i) continue;
            const float dd = sqrt_(norm2(z32[i] - z32[j]));
            num *= az + sqrt_(norm2(z32[j]));
            den *= dd;
            gap = fmin(gap, dd);
        }
        if (!((kNoise * 1.1102230e-16f) * num <= kTightRoots * den * gap)) return false;
    }
    cx<float> zi[5], wi[5];  // the images found
    int count = 0, parity = 0;
    bool fold = false;
    double sum = 0.0;
    cx<double> zs = mk<double>(0.0, 0.0), zp = mk<double>(1.0, 0.0);
    for (int i = 0; i < 5; ++i) {
        cx<double> z, w;
        start_from_fp32(z32[i], d, z, w);
        const Refined f = refine_root<false>(z, w, zeta, q, 8);
        if (!f.image) continue;
        const cx<float> zf = mk<float>((float)f.z.re, (float)f.z.im), wf = mk<float>((float)f.w.re, (float)f.w.im);
        bool dup = false;
        for (int j = 0; j < count; ++j)
            dup = dup || (norm2(zi[j] - zf) <= 1e-11f * fmin(norm2(zi[j]), norm2(zf)) &&
                          norm2(wi[j] - wf) <= 1e-11f * fmin(norm2(wi[j]), norm2(wf)));
        if (dup) continue;
        zi[count] = zf;
        wi[count] = wf;
        ++count;
        parity += f.det < 0.0 ? -1 : 1;
        const double a = fabs(f.det);
        fold = fold || (float)a < kFoldDet;
        sum += rcp_normal(a);
        zs = zs + f.z;
        zp = zp * f.z;
    }
    *A = sum;
    if (parity != -1 || fold) return false;
    if (count == 5) return true;
    return count == 3 && remaining_root_spurious(zs, zp, zeta, d, q, 0) &&
           remaining_root_spurious(zs, zp, zeta, d, q, 1);
}

}  // namespace sblm
