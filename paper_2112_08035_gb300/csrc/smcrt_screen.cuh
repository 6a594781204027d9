// smcrt_screen.cuh -- FP32 screening for the FP64 packet kernel.
//
// GB300 has one FP64 pipe per SM, which takes 16 cycles for a warp
// instruction: one FP64 operation costs as much issue time as 64 FP32 or
// integer ones.  The kernel's results must be the reference's IEEE
// operations on the values that count, but most values do not: the distance
// of a region that is not the nearest, the plane of an axis that the ray
// does not reach, a move's bound when the packet interacts before it.  Here
// FP32 arithmetic with a proven error bound finds out which values count,
// and only those are computed in FP64, by the reference's expressions.
// Wherever FP32 cannot tell, the FP64 code runs: results are bit-identical.
//
// Error bound.  Let R bound every coordinate, half extent and radius of the
// scene (bounding box, primitives, source) plus four surface thresholds,
// and u = 2^-24.  A packet stays within R of the origin on every axis.  The
// FP32 distance of a sphere or box has an error below 30 u R (rounded
// inputs 4 u R per component, a norm of up to 2 sqrt(3) R, two ulps of the
// square root), of a capsule below 80 u R (the foot point along the axis),
// and each of up to 8 smooth unions adds 14 u R (min, max and the
// polynomial smooth minimum are 1-Lipschitz in their operands, so operand
// errors do not grow).  DevScene.feps = 2^-16 R = 256 u R exceeds the sum.
#pragma once

#include "smcrt_kernel.cuh"

namespace smcrt {

constexpr float kScrUp = 1.00001f, kScrDown = 0.99999f;   // covers a few FP32 roundings of a product

__device__ __forceinline__ float scr_sqrt(float x) { return x * rsqrtf(fmaxf(x, 1e-30f)); }

__device__ __forceinline__ float scr_box(float x, float y, float z, float cx, float cy, float cz, float hx, float hy,
                                         float hz)
{
    const float qx = fabsf(x - cx) - hx, qy = fabsf(y - cy) - hy, qz = fabsf(z - cz) - hz;
    const float mx = fmaxf(qx, 0.f), my = fmaxf(qy, 0.f), mz = fmaxf(qz, 0.f);
    return scr_sqrt(__fmaf_rn(mx, mx, __fmaf_rn(my, my, mz * mz))) + fminf(fmaxf(qx, fmaxf(qy, qz)), 0.f);
}

__device__ __forceinline__ float scr_prim(const DevScene &S, int kind, int i, float x, float y, float z)
{
    const float4 A = __ldg(S.p32 + 2 * i);
    const float ax = x - A.x, ay = y - A.y, az = z - A.z;
    if (kind == 0) return scr_sqrt(__fmaf_rn(ax, ax, __fmaf_rn(ay, ay, az * az))) - A.w;
    const float4 B = __ldg(S.p32 + 2 * i + 1);
    if (kind == 1) return scr_box(x, y, z, A.x, A.y, A.z, B.x, B.y, B.z);
    const float t = __saturatef(__fmaf_rn(ax, B.x, __fmaf_rn(ay, B.y, az * B.z)) * B.w);
    const float dx = __fmaf_rn(-B.x, t, ax), dy = __fmaf_rn(-B.y, t, ay), dz = __fmaf_rn(-B.z, t, az);
    return scr_sqrt(__fmaf_rn(dx, dx, __fmaf_rn(dy, dy, dz * dz))) - A.w;
}

// A left fold of unions and smooth unions (one instruction per primitive).
// Where |acc - d| is certainly at least k, the smooth minimum's h is clamped
// to 0 or 1 and the FP64 fold returns the smaller operand exactly: a farther
// primitive leaves the fold as it is, a nearer one makes everything before it
// irrelevant.  What is left to fold in FP64 are the instructions since the
// last such reset that do not leave the fold alone: `list`, 16 bits each, in
// order; cnt > kFoldList: too many, all of them count.  Each blend of two
// operands adds 14 u R to the value's error; beyond the 8 that feps covers
// the bound grows with them (err).  On the 64-capsule vessel tree 1 to 3
// capsules are left of 64.
constexpr int kFoldList = 4;

__device__ __noinline__ float fold_screen(const DevScene &S, int i0, int i1, float x, float y, float z,
                                          unsigned long long &list, int &cnt, float &err)
{
    const float eps = S.feps;
    float acc = 0.f, ea = eps;
    unsigned long long li = 0ull;
    int n = 0;
    for (int i = i0; i < i1; ++i) {
        const int4 ins = __ldg(reinterpret_cast<const int4 *>(S.instr) + i);
        const int op = ins.x & 0xff;
        const float d = scr_prim(S, (ins.x >> 8) & 0xff, ins.y, x, y, z);
        const float kinv = __int_as_float(ins.w);
        const float gap = fabsf(acc - d) - (ea + eps);
        const bool sure = op == 2 ? gap * kinv > kScrUp : gap > 0.f;
        if (op == 0 || sure) {
            if (op == 0 || d < acc) {
                acc = d;
                ea = eps;
                li = (unsigned long long)(unsigned)(i - i0);
                n = 1;
            }
        } else {
            if (n < kFoldList) li |= (unsigned long long)(unsigned)(i - i0) << (16 * n);
            ++n;
            if (n > 9) ea = __fmaf_rn(eps, 1.f / 16.f, ea) * kScrUp;
            acc = op == 2 ? csg32(2, acc, d, kinv) : fminf(acc, d);
        }
    }
    list = li;
    cnt = n;
    err = ea;
    return acc;
}

// Any other region program in FP32 (at most 8 smooth unions).
static __device__ __noinline__ float prog_screen(const DevScene &S, int i0, int i1, float x, float y, float z)
{
    float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
    for (int i = i0; i < i1; ++i) {
        const int4 ins = __ldg(reinterpret_cast<const int4 *>(S.instr) + i);
        const int op = ins.x & 0xff;
        float v = 0.f;
        if (ins.y >= 0) v = scr_prim(S, (ins.x >> 8) & 0xff, ins.y, x, y, z);
        if (op == 0) {
            s3 = s2; s2 = s1; s1 = s0; s0 = v;
        } else if (ins.y >= 0) {
            s0 = csg32(op, s0, v, __int_as_float(ins.w));
        } else {
            s0 = csg32(op, s1, s0, __int_as_float(ins.w));
            s1 = s2; s2 = s3;
        }
    }
    return s0;
}

// The FP64 value of region r: of a fold the listed instructions (cnt >= 0), or
// the whole program.  Out of line, with the one copy of the primitives: code
// size counts (see div64).
static __device__ __noinline__ double region_exact(const DevScene &S, int r, double x, double y, double z,
                                                   unsigned long long list, int cnt)
{
    const int2 rr = __ldg(S.rrange + r);
    const bool listed = cnt >= 0 && cnt <= kFoldList;
    const int n = listed ? cnt : rr.y - rr.x;
    double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
    for (int k = 0; k < n; ++k) {
        const int i = rr.x + (listed ? (int)(list & 0xffffull) : k);
        list >>= 16;
        const int4 ins = __ldg(reinterpret_cast<const int4 *>(S.instr) + i);
        const int op = listed && k == 0 ? 0 : ins.x & 0xff;
        double v = 0.0;
        if (ins.y >= 0) v = prim64<false>(S, (ins.x >> 8) & 0xff, ins.y, x, y, z);
        if (op == 0) {
            s3 = s2; s2 = s1; s1 = s0; s0 = v;
        } else {
            const double a = ins.y >= 0 ? s0 : s1, b = ins.y >= 0 ? v : s0;
            if (ins.y < 0) { s1 = s2; s2 = s3; }
            s0 = csg64(op, a, b, op == 2 ? __ldg(S.k64 + i) : 0.0);
        }
    }
    return s0;
}

// The list of region r where it is a fold worth one (cnt = -1: none).
__device__ __forceinline__ void fold_list(const DevScene &S, int r, double x, double y, double z,
                                          unsigned long long &list, int &cnt)
{
    cnt = -1;
    list = 0ull;
    if (!((S.fold_mask >> r) & 1ull)) return;
    const int2 rr = __ldg(S.rrange + r);
    float err;
    if (rr.y - rr.x > kFoldList) fold_screen(S, rr.x, rr.y, (float)x, (float)y, (float)z, list, cnt, err);
}

// What an evaluation is for: a trace position (region, nearest surface), one
// surface's value (normal probes, projection), or the region at a point.
enum EvalFor { kForTrace = 0, kForSurface = 1, kForRegion = 2 };

// Scene evaluation in which only the values that count are FP64: the
// regions that may be nearest (trace), whose sign FP32 cannot tell, or the
// one surface asked for.  dsoft: a lower bound (FP32) over the soft regions;
// dbox: FP64 where it may be nearest, else an FP32 value of the right sign.
// Layered slab: 1.1 of 4 surfaces are left per trace evaluation; without the
// square root where at most one axis is outside (box_exact).
static __device__ __noinline__ Eval64 scene_eval64_screened(const DevScene &S, double x, double y, double z, int sel,
                                                        int mode)
{
    Eval64 E;
    E.dmin = __longlong_as_double(0x7ff0000000000000LL);
    E.dsoft = E.dmin;
    E.dstar = 0.0; E.dsel = 0.0; E.dbox = -1.0; E.istar = -1; E.region = -1;
    const float inf = __int_as_float(0x7f800000), eps = S.feps;
    const float fx = (float)x, fy = (float)y, fz = (float)z;
    unsigned long long neg = 0ull, mask = 0ull, list = 0ull;
    int flr = -1, cnt = 0;                       // the fold whose list is at hand
    float mlo = inf, mhi = inf, soft = inf;      // bounds of the smallest |d|
    if (mode == kForSurface) {
        if (sel >= 0) mask = 1ull << sel;
    } else {
        for (int r = 0; r < S.nregions; ++r) {
            const unsigned long long bit = 1ull << r;
            if (!(S.screen_mask & bit)) {        // FP32 says nothing about this one
                mask |= bit;
                if (S.soft_mask & bit) soft = 0.f;
                continue;
            }
            const int2 rr = __ldg(S.rrange + r);
            float d, err = eps;
            unsigned long long li = 0ull;
            int n = 0;
            if (S.fold_mask & bit) d = fold_screen(S, rr.x, rr.y, fx, fy, fz, li, n, err);
            else d = prog_screen(S, rr.x, rr.y, fx, fy, fz);
            if (d < 0.f) neg |= bit;
            const float lo = fabsf(d) - err, hi = fabsf(d) + err;
            if (S.soft_mask & bit) soft = fminf(soft, lo);
            bool in;
            if (mode == kForRegion) {
                in = !(lo > 0.f);
            } else {
                in = !(lo > mhi);
                if (hi < mlo) {                  // nearer than all so far: they are out
                    mask &= ~S.screen_mask;
                    mlo = lo;
                } else if (in) {
                    mlo = fminf(mlo, lo);
                }
                mhi = fminf(mhi, hi);
            }
            if (in) {
                mask |= bit;
                if (S.fold_mask & bit) { flr = r; list = li; cnt = n; }
            }
        }
    }
    while (mask != 0ull) {
        const int r = __ffsll((long long)mask) - 1;
        const unsigned long long bit = 1ull << r;
        mask ^= bit;
        unsigned long long li = list;
        int n = cnt;
        if (r != flr) fold_list(S, r, x, y, z, li, n);
        const double d = region_exact(S, r, x, y, z, li, n);
        if (d < 0.0) neg |= bit; else neg &= ~bit;
        const double ad = fabs(d);
        if (less64(ad, E.dmin)) { E.dmin = ad; E.istar = r; E.dstar = d; }
        if (r == sel) E.dsel = d;
    }
    if (neg != 0ull) E.region = 63 - __clzll((long long)neg);
    E.dsoft = (double)soft;
    const float db = mode == kForTrace ? scr_box(fx, fy, fz, S.bbc32[0], S.bbc32[1], S.bbc32[2], S.bbh32[0],
                                                 S.bbh32[1], S.bbh32[2])
                                       : 0.f;
    if (mode == kForTrace) E.dbox = (double)db;
    if ((mode == kForTrace && (!(fabsf(db) - eps > mhi) || !(fabsf(db) > eps))) || (mode == kForSurface && sel == -1)) {
        const double d = box64(x, y, z, S.bbc[0], S.bbc[1], S.bbc[2], S.bbh[0], S.bbh[1], S.bbh[2]);
        E.dbox = d;
        if (fabs(d) < E.dmin) { E.dmin = fabs(d); E.istar = -1; E.dstar = d; }
        if (sel == -1) E.dsel = d;
    }
    return E;
}

// A packet within delta of a surface (Sec. 2.3), all of it at once: the
// normal by central differences, the approach test, the projection and the
// regions on both sides.  A warp's packets that have arrived wait until
// several have (k64: kArrive), instead of taking one of these ten or so
// evaluations per loop iteration while the other lanes tally and scatter.
struct Interface64 {
    double nx, ny, nz, qx, qy, qz, cdot, n1, n2, ct, R;
    int what;                // see below
    int evals;               // scene evaluations
};
enum { kIntfForced = 0, kIntfEscape = 1, kIntfMatched = 2, kIntfFresnel = 3 };

template <bool G>
static __device__ __noinline__ double surface_at64(const DevScene &S, int r, double x, double y, double z)
{
    if (G || r < 0) return surface64<G>(S, r, x, y, z);
    unsigned long long list = 0ull;
    int cnt;
    fold_list(S, r, x, y, z, list, cnt);
    return region_exact(S, r, x, y, z, list, cnt);
}

template <bool G>
static __device__ __noinline__ int region_at64(const DevScene &S, double x, double y, double z)
{
    return (G ? scene_eval64<G>(S, x, y, z, -2) : scene_eval64_screened(S, x, y, z, -2, kForRegion)).region;
}

__device__ __forceinline__ double region_n64(const DevScene &S, int r)
{
    return r < 0 ? S.ambient_n : __ldg(S.reg64 + 8 * r + 3);
}

template <bool G>
static __device__ __noinline__ Interface64 interface64(const DevScene &S, double px, double py, double pz, double ux,
                                                       double uy, double uz, int istar, double dstar)
{
    const double delta = S.delta;
    Interface64 o;
    o.what = kIntfForced;
    o.evals = 6;
    o.R = 1.0; o.ct = 0.0;
    o.cdot = 0.0;
    double gx = 0.0, gy = 0.0, gz = 0.0;
    for (int a = 0; a < 3; ++a) {            // central differences
        const double ex = a == 0 ? delta : 0.0, ey = a == 1 ? delta : 0.0, ez = a == 2 ? delta : 0.0;
        const double fp = surface_at64<G>(S, istar, px + ex, py + ey, pz + ez);
        const double fm = surface_at64<G>(S, istar, px - ex, py - ey, pz - ez);
        gx = gy; gy = gz; gz = fp - fm;      // after three turns: x, y, z
    }
    const double l2 = gx * gx + gy * gy + gz * gz;
    if (!(l2 > 0.0)) return o;
    const double l = sqrt64(l2);
    const double nx = div64(gx, l), ny = div64(gy, l), nz = div64(gz, l);
    const double cdot = ux * nx + uy * ny + uz * nz;
    o.nx = nx; o.ny = ny; o.nz = nz;
    o.cdot = cdot;
    if (!((cdot > 0.0 && dstar < 0.0) || (cdot < 0.0 && dstar >= 0.0))) return o;
    o.what = kIntfEscape;
    if (istar < 0) return o;
    double qx = px, qy = py, qz = pz;        // Newton projection
    for (int k = 0; k < 3; ++k) {
        const double dq = surface_at64<G>(S, istar, qx, qy, qz);
        o.evals += 1;
        if (fabs(dq) <= delta * 1e-3) break;
        qx = qx - dq * nx; qy = qy - dq * ny; qz = qz - dq * nz;
    }
    o.qx = qx; o.qy = qy; o.qz = qz;
    const double ee = 2.0 * delta * (cdot > 0.0 ? 1.0 : -1.0);
    o.n2 = region_n64(S, region_at64<G>(S, qx + ee * nx, qy + ee * ny, qz + ee * nz));
    o.n1 = region_n64(S, region_at64<G>(S, qx - ee * nx, qy - ee * ny, qz - ee * nz));
    o.evals += 2;
    o.what = kIntfMatched;
    if (o.n1 == o.n2) return o;
    o.what = kIntfFresnel;
    const double n1 = o.n1, n2 = o.n2, ci = fabs(cdot);
    const double eta = div64(n1, n2);
    const double st2 = eta * eta * ((1.0 - ci) * (1.0 + ci));
    if (st2 < 1.0) {
        const double ct = sqrt64(1.0 - st2);
        const double rs = div64(n1 * ci - n2 * ct, n1 * ci + n2 * ct);
        const double rp = div64(n1 * ct - n2 * ci, n1 * ct + n2 * ci);
        o.ct = ct;
        o.R = 0.5 * (rs * rs + rp * rp);
    }
    return o;
}

// ---------------------------------------------------------------------------
// Segment stepping
// ---------------------------------------------------------------------------

// FP32 ray against a box (half extents h): lower bounds of the exit from
// inside and of the entry from outside (inf: certainly missed).
__device__ __forceinline__ float scr_exit(float c, float h, float p, float u, float eps)
{
    const float d = h - (u > 0.f ? p - c : c - p) - eps;
    return u == 0.f ? __int_as_float(0x7f800000) : d > 0.f ? __fdividef(d, fabsf(u)) * kScrDown : 0.f;
}

__device__ __forceinline__ float scr_box_exit(const float *c, const float *h, float e, const float *p, const float *u,
                                              float eps)
{
    return fminf(scr_exit(c[0], h[0] - e, p[0], u[0], eps),
                 fminf(scr_exit(c[1], h[1] - e, p[1], u[1], eps), scr_exit(c[2], h[2] - e, p[2], u[2], eps)));
}

__device__ __forceinline__ float scr_box_entry(const float *c, const float *h, float e, const float *p, const float *u,
                                               float eps)
{
    const float inf = __int_as_float(0x7f800000);
    float tn = 0.f, tf = inf;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float q = u[a] > 0.f ? p[a] - c[a] : c[a] - p[a], g = h[a] + e;
        const float in = -g - q - eps, out = g - q + eps;    // along the ray, lower / upper
        if (u[a] == 0.f) {
            if (fabsf(q) > g + eps) return inf;
            continue;
        }
        const float iu = __fdividef(1.f, fabsf(u[a]));
        if (out < 0.f) return inf;
        tf = fminf(tf, out * iu * kScrUp);
        if (in > 0.f) tn = fmaxf(tn, in * iu * kScrDown);
    }
    return tn > tf ? inf : tn;
}

// FP32 ray against a sphere: the same two bounds.  The discriminant's error
// is below 64 u times the sum of its terms.
__device__ __forceinline__ float scr_sphere(float4 A, float d, float e, const float *p, const float *u, float eps)
{
    const float rr = d > 0.f ? A.w + e : A.w - e;
    const float ox = p[0] - A.x, oy = p[1] - A.y, oz = p[2] - A.z;
    const float b = ox * u[0] + oy * u[1] + oz * u[2];
    const float oo = ox * ox + oy * oy + oz * oz;
    const float err = 4e-6f * (oo + rr * rr + b * b) + 2.f * eps * (fabsf(b) + scr_sqrt(oo) + rr);
    const float disc = b * b - oo + rr * rr;
    if (d > 0.f) {
        if (b > eps || disc + err < 0.f) return __int_as_float(0x7f800000);
        return -b - scr_sqrt(fmaxf(disc + err, 0.f)) * kScrUp - eps;
    }
    if (disc - err < 0.f) return 0.f;
    return scr_sqrt(disc - err) * kScrDown - b - eps;
}

// A lower bound of the move bound (segment_bound64), or a value <= 0 when
// FP32 cannot tell.
static __device__ __noinline__ float segment_screen(const DevScene &S, float soft, const float *p, const float *u)
{
    const float eps = S.feps, dh = (float)(0.5 * S.delta) * kScrUp;
    if (eps == 0.f) return 0.f;
    float t = fminf(scr_box_exit(S.bbc32, S.bbh32, dh, p, u, eps), soft - dh);
    for (int j = 0; j < S.nseg; ++j) {
        const int i = __ldg(S.seg_prims + j), kind = __ldg(S.pkind + i);
        const float e = __ldg(S.seg_m32 + j) * kScrUp + dh;
        const float d = scr_prim(S, kind, i, p[0], p[1], p[2]);
        float b = fabsf(d) - eps - e;
        if (!(b > 0.f)) return 0.f;
        if (b >= t) continue;
        const float4 A = __ldg(S.p32 + 2 * i), B = __ldg(S.p32 + 2 * i + 1);
        const float c[3] = {A.x, A.y, A.z}, h[3] = {B.x, B.y, B.z};
        if (kind == 1) b = fmaxf(b, d > 0.f ? scr_box_entry(c, h, e, p, u, eps) : scr_box_exit(c, h, e, p, u, eps));
        else if (kind == 0) b = fmaxf(b, scr_sphere(A, d, e, p, u, eps));
        t = fminf(t, b);
    }
    return t;
}

// Exit from inside a box shrunk by e, where FP32 finds the axes that may come
// first and only their quotients are taken (the reference takes the larger of
// an axis' two quotients, which is the one of the plane ahead: rounding is
// monotone).
static __device__ __noinline__ double seg_exit64(double cx, double cy, double cz, double hx, double hy, double hz,
                                             double d, double px, double py, double pz, double ux, double uy,
                                             double uz, double e, float eps)
{
    const double c[3] = {cx, cy, cz}, h[3] = {hx, hy, hz}, p[3] = {px, py, pz}, u[3] = {ux, uy, uz};
    float lo[3], first = __int_as_float(0x7f800000);
    bool odd = false;                        // a direction component of zero, a box thinner than 2 e
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float uf = (float)u[a], hf = (float)h[a] - (float)e;
        const float q = uf > 0.f ? (float)p[a] - (float)c[a] : (float)c[a] - (float)p[a];
        odd = odd || uf == 0.f || !(hf > eps);
        const float iu = __fdividef(1.f, fabsf(uf));
        lo[a] = fmaxf(hf - q - eps, 0.f) * iu * kScrDown;
        first = fminf(first, fmaxf(hf - q + eps, 0.f) * iu * kScrUp);
    }
    if (eps == 0.f || odd || !(first < 1e30f)) return seg_box64(cx, cy, cz, hx, hy, hz, d, px, py, pz, ux, uy, uz, e);
    double tf = __longlong_as_double(0x7ff0000000000000LL);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (lo[a] > first) continue;
        const double he = h[a] + (-e);
        tf = fmin(tf, div64((u[a] > 0.0 ? c[a] + he : c[a] - he) - p[a], u[a]));
    }
    return tf > 0.0 ? tf : 0.0;
}

// The move bound of segment_bound64, leaving out what cannot lower it.
static __device__ __noinline__ double segment_bound64_screened(const DevScene &S, double soft, double dbox, double px,
                                                               double py, double pz, double ux, double uy, double uz)
{
    const float eps = S.feps;
    const float p[3] = {(float)px, (float)py, (float)pz}, u[3] = {(float)ux, (float)uy, (float)uz};
    const double dh = 0.5 * S.delta;
    double t = dbox > 0.0 ? seg_box64(S.bbc[0], S.bbc[1], S.bbc[2], S.bbh[0], S.bbh[1], S.bbh[2], dbox, px, py, pz,
                                      ux, uy, uz, dh)
                          : seg_exit64(S.bbc[0], S.bbc[1], S.bbc[2], S.bbh[0], S.bbh[1], S.bbh[2], dbox, px, py, pz,
                                       ux, uy, uz, dh, eps);
    if (S.soft_mask != 0ull && soft - dh <= t) {
        double ds = __longlong_as_double(0x7ff0000000000000LL);
        for (unsigned long long m = S.soft_mask; m != 0ull; m &= m - 1ull) {
            const int r = __ffsll((long long)m) - 1;
            unsigned long long list = 0ull;
            int cnt;
            fold_list(S, r, px, py, pz, list, cnt);
            ds = fmin(ds, fabs(region_exact(S, r, px, py, pz, list, cnt)));
        }
        t = fmin(t, ds - dh);
    }
    for (int j = 0; j < S.nseg; ++j) {
        const int i = __ldg(S.seg_prims + j);
        const int kind = __ldg(S.pkind + i);
        const double e = __ldg(S.seg_m64 + j) + dh;
        const float ef = (float)e * kScrUp, tu = (float)t * kScrUp;
        const float df = scr_prim(S, kind, i, p[0], p[1], p[2]);
        const float iso = fabsf(df) - eps - ef;
        const float4 A = __ldg(S.p32 + 2 * i), B = __ldg(S.p32 + 2 * i + 1);
        const float c[3] = {A.x, A.y, A.z}, h[3] = {B.x, B.y, B.z};
        if (eps > 0.f && iso > 0.f) {        // certainly outside the margin
            if (iso > tu) continue;
            if (kind == 1 &&
                (df > 0.f ? scr_box_entry(c, h, ef, p, u, eps) : scr_box_exit(c, h, ef, p, u, eps)) > tu)
                continue;
            if (kind == 0 && scr_sphere(A, df, ef, p, u, eps) > tu) continue;
        }
        const double d = prim64<false>(S, kind, i, px, py, pz);
        if (!(fabs(d) > e)) return 0.0;
        if (fabs(d) - e >= t) continue;
        const double *P = S.p64 + 8 * i;
        double b;
        if (kind == 0)
            b = seg_sphere64(P, d, px, py, pz, ux, uy, uz, e);
        else if (kind == 1)
            b = d > 0.0 ? seg_box64(__ldg(P), __ldg(P + 1), __ldg(P + 2), __ldg(P + 3), __ldg(P + 4), __ldg(P + 5), d,
                                    px, py, pz, ux, uy, uz, e)
                        : seg_exit64(__ldg(P), __ldg(P + 1), __ldg(P + 2), __ldg(P + 3), __ldg(P + 4), __ldg(P + 5),
                                     d, px, py, pz, ux, uy, uz, e, eps);
        else
            b = seg_capsule64(P, d, px, py, pz, ux, uy, uz, e);
        t = fmin(t, b);
    }
    return t;
}

// ---------------------------------------------------------------------------
// Track-length tally: tally64 with the grid clip left out where the segment
// starts inside the grid, the voxel index taken from FP32 where its fraction
// is clear of a voxel boundary, and one plane's quotient taken per voxel
// crossing (the axis that certainly comes first) in place of three and of a
// comparison of three.  Positions are in voxels from the grid's corner (one
// FP64 subtraction per axis); the FP32 error of one is below
// DevScene.gm32 = 16 u n.  A segment inside one voxel (most of them) takes
// five FP64 operations, a crossing 16.
// ---------------------------------------------------------------------------
static __device__ __noinline__ unsigned tally64_screened(const DevScene &S, long long *flu, double px, double py,
                                                         double pz, double ux, double uy, double uz, double len,
                                                         double w)
{
    if (!(len > 0.0) || !(w > 0.0)) return 0u;
    const float lf = (float)len;
    const float mx = S.gm32[0], my = S.gm32[1], mz = S.gm32[2];
    const int nx = S.g_n[0], ny = S.g_n[1], nz = S.g_n[2];
    const float gx = (float)(px - S.g_lo[0]) * S.g_idl32[0], ax = lf * (float)ux * S.g_idl32[0], hx = gx + ax;
    const float gy = (float)(py - S.g_lo[1]) * S.g_idl32[1], ay = lf * (float)uy * S.g_idl32[1], hy = gy + ay;
    const float gz = (float)(pz - S.g_lo[2]) * S.g_idl32[2], az = lf * (float)uz * S.g_idl32[2], hz = gz + az;
    // both ends beyond one side of the grid: no voxel
    const float ex = mx + 1e-6f * (fabsf(gx) + fabsf(ax)), ey = my + 1e-6f * (fabsf(gy) + fabsf(ay)),
                ez = mz + 1e-6f * (fabsf(gz) + fabsf(az));
    if (fminf(gx, hx) > (float)nx + ex || fmaxf(gx, hx) < -ex || fminf(gy, hy) > (float)ny + ey ||
        fmaxf(gy, hy) < -ey || fminf(gz, hz) > (float)nz + ez || fmaxf(gz, hz) < -ez)
        return 0u;
    const float bx = floorf(gx), by = floorf(gy), bz = floorf(gz);
    float sx = gx - bx, sy = gy - by, sz = gz - bz;          // position in the voxel
    const bool clear = gx > mx && gx < (float)nx - mx && gy > my && gy < (float)ny - my && gz > mz &&
                       gz < (float)nz - mz && fminf(sx, 1.f - sx) > 2.f * mx && fminf(sy, 1.f - sy) > 2.f * my &&
                       fminf(sz, 1.f - sz) > 2.f * mz;
    if (!clear) return tally64(S, flu, px, py, pz, ux, uy, uz, len, w);
    int ix = (int)bx, iy = (int)by, iz = (int)bz;
    // voxels to the plane ahead of each axis, and 1 / (voxels the segment advances)
    sx = ax > 0.f ? 1.f - sx : sx; sy = ay > 0.f ? 1.f - sy : sy; sz = az > 0.f ? 1.f - sz : sz;
    const float vx = __fdividef(1.f, fmaxf(fabsf(ax), 1e-30f)), vy = __fdividef(1.f, fmaxf(fabsf(ay), 1e-30f)),
                vz = __fdividef(1.f, fmaxf(fabsf(az), 1e-30f));
    double t = 0.0;
    unsigned npieces = 0u;
    for (;;) {
        // where the planes ahead lie along the segment (1 = its end)
        const float lx = (sx - 2.f * mx) * vx * kScrDown, ly = (sy - 2.f * my) * vy * kScrDown,
                    lz = (sz - 2.f * mz) * vz * kScrDown;
        const bool ends = fminf(lx, fminf(ly, lz)) > kScrUp;  // in this voxel
        const float ox = (sx + 2.f * mx) * vx * kScrUp, oy = (sy + 2.f * my) * vy * kScrUp,
                    oz = (sz + 2.f * mz) * vz * kScrUp;
        const bool cx = ox < fminf(ly, lz), cy = oy < fminf(lx, lz), cz = oz < fminf(lx, ly);
        if (!ends && (!(cx || cy || cz) || !(fminf(ox, fminf(oy, oz)) < kScrDown)))   // a tie, for FP32
            return npieces + walk64(S, flu, px, py, pz, ux, uy, uz, ix, iy, iz, t, len, w);
        const bool up = (cx ? ax : cy ? ay : az) > 0.f;
        const int i = cx ? ix : cy ? iy : iz, n = cx ? nx : cy ? ny : nz;
        const bool leaves = !ends && (up ? i + 1 >= n : i == 0);
        double tend = len;
        if (!ends) {
            const double lo = cx ? S.g_lo[0] : cy ? S.g_lo[1] : S.g_lo[2];
            const double dl = cx ? S.g_dl[0] : cy ? S.g_dl[1] : S.g_dl[2];
            const double p = cx ? px : cy ? py : pz, u = cx ? ux : cy ? uy : uz;
            tend = div64((lo + (double)(i + up) * dl) - p, u);
            if (leaves) {                        // the grid's own face clips the segment
                const double hi = cx ? S.g_hi[0] : cy ? S.g_hi[1] : S.g_hi[2];
                tend = fmin(tend, div64((up ? hi : lo) - p, u));
            }
        }
        const double piece = tend - t;
        if (piece > 0.0) {
            red_add(flu + ((long long)iz * ny + iy) * nx + ix, fx64(w * piece));
            npieces += 1u;
            t = tend;
        }
        if (ends || leaves) return npieces;
        const int s = up ? 1 : -1;
        if (cx) { ix += s; sx += 1.f; }
        else if (cy) { iy += s; sy += 1.f; }
        else { iz += s; sz += 1.f; }
    }
}

}  // namespace smcrt
