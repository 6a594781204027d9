// smcrt_screen.cuh -- FP32 screening for the FP64 packet kernel.
//
// An FP64 warp instruction takes a scheduler of GB300 64 cycles (measured; an
// SM's four schedulers start one every 16 cycles between them, 19 with all at
// it): as much issue time as 64 FP32 or integer ones.  The kernel's results must be the reference's IEEE
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
// errors do not grow).  DevScene.feps exceeds the sum: 2^-16 R = 256 u R, and in
// scenes of simple regions a few delta more (segment_bound64_screened).
#pragma once

#include <cstddef>

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
// capsules are left of 64.  A packet's turn through the loop waits for the 64
// distances one after the other, each a chain of about 100 cycles; in tree
// scenes, whose folds hold capsules only, four are computed side by side
// (without a branch on the kind in between, which kept the compiler from it):
// vessel tree 1e4 packets 53.1 -> 36.2 ms with the other shapes left out; 39.7
// with eight.
constexpr int kFoldList = 4;

template <int K>
static __device__ __noinline__ float fold_screen(const DevScene &S, int i0, int i1, float x, float y, float z,
                                                 float slack, unsigned long long &list, int &cnt, float &err)
{
    const float eps = S.feps + slack;
    float acc = 0.f, ea = eps;
    unsigned long long li = 0ull;
    int n = 0;
    constexpr int kAhead = K == kTreeScene ? 4 : 1;
    for (int b = i0; b < i1; b += kAhead) {
        int4 ins[kAhead];
        float ds[kAhead];
#pragma unroll
        for (int k = 0; k < kAhead; ++k) ins[k] = __ldg(reinterpret_cast<const int4 *>(S.instr) + min(b + k, i1 - 1));
#pragma unroll
        for (int k = 0; k < kAhead; ++k)
            ds[k] = scr_prim(S, K == kTreeScene ? 2 : (ins[k].x >> 8) & 0xff, ins[k].y, x, y, z);
#pragma unroll
        for (int k = 0; k < kAhead; ++k) {
            const int i = b + k;
            if (i >= i1) break;
            const int op = ins[k].x & 0xff;
            const float d = ds[k];
            const float kinv = __int_as_float(ins[k].w);
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

// The functions below are instantiated per scene family (K), as the kernels.
template <int K>
__device__ constexpr bool one_each()     // one primitive per region
{
    return K == kBoxScene || K == kSingleScene;
}

// The FP64 value of region r: of a fold the listed instructions (cnt >= 0), or
// the whole program.  Out of line, with the one copy of the primitives: code
// size counts (see div64).
template <int K>
static __device__ __noinline__ double region_exact(const DevScene &S, int r, double x, double y, double z,
                                                   unsigned long long list, int cnt)
{
    const int2 rr = __ldg(S.rrange + r);
    if (one_each<K>()) {                 // its one primitive
        const int4 ins = __ldg(reinterpret_cast<const int4 *>(S.instr) + rr.x);
        return base64<false>(K == kBoxScene ? 1 : (ins.x >> 8) & 0xff, S.p64 + 8 * ins.y, x, y, z);
    }
    if (K == kTreeScene && rr.y - rr.x == 1) {   // a box
        const int4 ins = __ldg(reinterpret_cast<const int4 *>(S.instr) + rr.x);
        return base64<false>(1, S.p64 + 8 * ins.y, x, y, z);
    }
    const bool listed = cnt >= 0 && cnt <= kFoldList;
    const int n = listed ? cnt : rr.y - rr.x;
    double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
    for (int k = 0; k < n; ++k) {
        const int i = rr.x + (listed ? (int)(list & 0xffffull) : k);
        list >>= 16;
        const int4 ins = __ldg(reinterpret_cast<const int4 *>(S.instr) + i);
        const int op = listed && k == 0 ? 0 : ins.x & 0xff;
        double v = 0.0;
        if (K == kTreeScene || ins.y >= 0) v = prim64<false>(S, K == kTreeScene ? 2 : (ins.x >> 8) & 0xff, ins.y, x, y, z);
        if (op == 0) {
            s3 = s2; s2 = s1; s1 = s0; s0 = v;
        } else {
            const double a = K == kTreeScene || ins.y >= 0 ? s0 : s1, b = K == kTreeScene || ins.y >= 0 ? v : s0;
            if (K != kTreeScene && ins.y < 0) { s1 = s2; s2 = s3; }
            s0 = csg64(op, a, b, op == 2 ? __ldg(S.k64 + i) : 0.0);
        }
    }
    return s0;
}

// The list of region r where it is a fold worth one (cnt = -1: none), good at
// all points within slack (distances and folds are 1-Lipschitz).
template <int K>
__device__ __forceinline__ void fold_list(const DevScene &S, int r, double x, double y, double z,
                                          float slack, unsigned long long &list, int &cnt)
{
    cnt = -1;
    list = 0ull;
    if (one_each<K>() || !((S.fold_mask >> r) & 1ull)) return;
    const int2 rr = __ldg(S.rrange + r);
    float err;
    if (rr.y - rr.x > kFoldList) fold_screen<K>(S, rr.x, rr.y, (float)x, (float)y, (float)z, slack, list, cnt, err);
}

// What an evaluation is for: a trace position (region, nearest surface) or the
// region at a point.
enum EvalFor { kForTrace = 0, kForRegion = 1 };

// The scene in FP32.
struct Screen64 {
    unsigned long long neg;  // regions with a negative value
    unsigned long long mask; // regions whose FP64 value counts (nearest, sign, or unscreened)
    unsigned long long list; // the list of fold flr, cnt entries
    int flr, cnt;
    float soft;              // lower bound of |d| over the soft regions
    float lo;                // lower bound of |d| over all surfaces; <= 0: some sign is open
    float db;                // bounding box
};

template <int K>
static __device__ __noinline__ Screen64 scene_screen(const DevScene &S, float x, float y, float z, int mode,
                                                     int flr = -1, unsigned long long list = 0ull, int cnt = 0)
{
    Screen64 C;
    const float inf = __int_as_float(0x7f800000), eps = S.feps;
    C.neg = C.mask = C.list = 0ull;
    C.flr = -1; C.cnt = 0;
    float mlo = inf, mhi = inf, soft = inf, all = inf;   // bounds of the smallest |d|
    for (int r = 0; r < S.nregions; ++r) {
        const unsigned long long bit = 1ull << r;
        if (!(S.screen_mask & bit)) {            // FP32 says nothing about this one
            C.mask |= bit;
            if (S.soft_mask & bit) soft = 0.f;
            all = -1.f;
            continue;
        }
        if (mode == kForRegion && r == flr) {    // a list is known already: straight to FP64
            C.mask |= bit;
            C.flr = r; C.list = list; C.cnt = cnt;
            all = -1.f;
            continue;
        }
        const int2 rr = __ldg(S.rrange + r);
        float d, err = eps;
        unsigned long long li = 0ull;
        int n = 0;
        if (one_each<K>() || (K == kTreeScene && rr.y - rr.x == 1)) {
            const int4 ins = __ldg(reinterpret_cast<const int4 *>(S.instr) + rr.x);
            d = scr_prim(S, K == kBoxScene || K == kTreeScene ? 1 : (ins.x >> 8) & 0xff, ins.y, x, y, z);
        } else if (K == kTreeScene || (S.fold_mask & bit)) {
            d = fold_screen<K>(S, rr.x, rr.y, x, y, z, 0.f, li, n, err);
        } else {
            d = prog_screen(S, rr.x, rr.y, x, y, z);
        }
        if (d < 0.f) C.neg |= bit;
        const float lo = fabsf(d) - err, hi = fabsf(d) + err;
        if (S.soft_mask & bit) soft = fminf(soft, lo);
        all = fminf(all, lo);
        bool in;
        if (mode == kForRegion) {
            in = !(lo > 0.f);
        } else {
            in = !(lo > mhi);
            if (hi < mlo) {                      // nearer than all so far: they are out
                C.mask &= ~S.screen_mask;
                mlo = lo;
            } else if (in) {
                mlo = fminf(mlo, lo);
            }
            mhi = fminf(mhi, hi);
        }
        if (in) {
            C.mask |= bit;
        }
        if (!one_each<K>() && (S.fold_mask & bit) && (mode == kForTrace ? in || C.flr < 0 : in && flr < 0)) {
            C.flr = r;
            C.list = li;
            C.cnt = min(n, kFoldList + 1);
        }
    }
    C.soft = soft;
    const float db = scr_box(x, y, z, S.bbc32[0], S.bbc32[1], S.bbc32[2], S.bbh32[0], S.bbh32[1], S.bbh32[2]);
    // db = 0: the box's FP64 value counts (it may be nearest, or its sign is open)
    C.db = !(fabsf(db) - eps > mhi) || !(fabsf(db) > eps) ? 0.f : db;
    C.lo = eps > 0.f ? fminf(all, -db - eps) : -1.f;
    return C;
}

// The scene evaluation from its screening, in which only the values that
// count are FP64.  dsoft: a lower bound (FP32) over the soft regions; dbox:
// FP64 where it may be nearest, else an FP32 value of the right sign.  1.1
// of the layered slab's 4 surfaces are left per trace evaluation, and no
// square root where at most one axis is outside (box64).
template <int K>
static __device__ __noinline__ Eval64 scene_exact(const DevScene &S, double x, double y, double z, const Screen64 &C,
                                                  int mode)
{
    Eval64 E;
    E.dmin = __longlong_as_double(0x7ff0000000000000LL);
    E.dstar = 0.0; E.istar = -1; E.region = -1;
    E.dsoft = (double)C.soft;
    E.dbox = (double)C.db;
    unsigned long long neg = C.neg, mask = C.mask;
    while (mask != 0ull) {
        const int r = __ffsll((long long)mask) - 1;
        const unsigned long long bit = 1ull << r;
        mask ^= bit;
        unsigned long long li = C.list;
        int n = C.cnt;
        if (!one_each<K>() && r != C.flr) fold_list<K>(S, r, x, y, z, 0.f, li, n);
        const double d = region_exact<K>(S, r, x, y, z, li, n);
        if (d < 0.0) neg |= bit; else neg &= ~bit;
        const double ad = fabs(d);
        if (less64(ad, E.dmin)) { E.dmin = ad; E.istar = r; E.dstar = d; }
    }
    if (neg != 0ull) E.region = 63 - __clzll((long long)neg);
    if (mode == kForTrace && C.db == 0.f) {
        const double d = box64(x, y, z, S.bbc[0], S.bbc[1], S.bbc[2], S.bbh[0], S.bbh[1], S.bbh[2]);
        E.dbox = d;
        if (less64(fabs(d), E.dmin)) { E.dmin = fabs(d); E.istar = -1; E.dstar = d; }
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

// A surface near a point where its fold list was made with a slack (cnt = -1:
// no list).  One screening of the fold for an interface's ten or so
// evaluations: vessel tree 1e4 packets 36.2 -> 35.2 ms, 4e4 56.5 -> 54.6.
struct FoldNear {
    unsigned long long list;
    int cnt;
};

template <int K>
static __device__ __noinline__ double surface_at64(const DevScene &S, int r, double x, double y, double z,
                                                   FoldNear f)
{
    if (K == kGeneralScene || r < 0) return surface64<K == kGeneralScene>(S, r, x, y, z);
    return region_exact<K>(S, r, x, y, z, f.list, f.cnt);
}

template <int K>
static __device__ __noinline__ int region_at64(const DevScene &S, double x, double y, double z, int r, FoldNear f)
{
    if (K == kGeneralScene) return scene_eval64(S, x, y, z).region;
    const Screen64 C = scene_screen<K>(S, (float)x, (float)y, (float)z, kForRegion, f.cnt >= 0 ? r : -1, f.list, f.cnt);
    return scene_exact<K>(S, x, y, z, C, kForRegion).region;
}

__device__ __forceinline__ double region_n64(const DevScene &S, int r)
{
    return r < 0 ? S.ambient_n : __ldg(S.reg64 + kReg64 * r + 3);
}

template <int K>
static __device__ __noinline__ Interface64 interface64(const DevScene &S, double px, double py, double pz, double ux,
                                                       double uy, double uz, int istar, double dstar)
{
    const double delta = S.delta;
    Interface64 o;
    o.what = kIntfForced;
    o.evals = 6;
    o.R = 1.0; o.ct = 0.0;
    o.cdot = 0.0;
    // one list for all the evaluations, within 6 delta: probes at delta, the
    // projection's steps (their sum is watched), the sides at 2 delta from it
    FoldNear f = {0ull, -1};
    if (K != kGeneralScene && istar >= 0) fold_list<K>(S, istar, px, py, pz, 6.f * (float)delta, f.list, f.cnt);
    double gx = 0.0, gy = 0.0, gz = 0.0;
    for (int a = 0; a < 3; ++a) {            // central differences
        const double ex = a == 0 ? delta : 0.0, ey = a == 1 ? delta : 0.0, ez = a == 2 ? delta : 0.0;
        const double fp = surface_at64<K>(S, istar, px + ex, py + ey, pz + ez, f);
        const double fm = surface_at64<K>(S, istar, px - ex, py - ey, pz - ez, f);
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
    float moved = 0.f;
    for (int k = 0; k < 3; ++k) {
        const double dq = surface_at64<K>(S, istar, qx, qy, qz, f);
        o.evals += 1;
        if (fabs(dq) <= delta * 1e-3) break;
        qx = qx - dq * nx; qy = qy - dq * ny; qz = qz - dq * nz;
        moved += fabsf((float)dq);
        if (K != kGeneralScene && moved > 3.9f * (float)delta) {   // too far for the list
            fold_list<K>(S, istar, qx, qy, qz, 6.f * (float)delta, f.list, f.cnt);
            moved = 0.f;
        }
    }
    o.qx = qx; o.qy = qy; o.qz = qz;
    const double ee = 2.0 * delta * (cdot > 0.0 ? 1.0 : -1.0);
    o.n2 = region_n64(S, region_at64<K>(S, qx + ee * nx, qy + ee * ny, qz + ee * nz, istar, f));
    o.n1 = region_n64(S, region_at64<K>(S, qx - ee * nx, qy - ee * ny, qz - ee * nz, istar, f));
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

// A lower bound of the distance along any ray to a primitive grown (d > 0) or
// shrunk by e, |d| known within eps: |d| - e, but a box grows by e with sharp
// corners, whose points lie up to sqrt(3) e from it.  Where every box's e is
// delta / 2 (scenes of simple regions), feps has room for that (fill_screen).
template <int K>
__device__ __forceinline__ float scr_isotropic(int kind, float d, float e, float eps)
{
    return fabsf(d) - eps - (K == kPlainScene && kind == 1 && d > 0.f ? 1.7321f * e : e);
}

// A lower bound of the move bound (segment_bound64), or a value <= 0 when
// FP32 cannot tell.
template <int K>
static __device__ __noinline__ float segment_screen(const DevScene &S, float soft, const float *p, const float *u)
{
    const float eps = S.feps, dh = (float)(0.5 * S.delta) * kScrUp;
    if (eps == 0.f) return 0.f;
    float t = fminf(scr_box_exit(S.bbc32, S.bbh32, dh, p, u, eps), soft - dh);
    for (int j = 0; j < S.nseg; ++j) {
        const int i = __ldg(S.seg_prims + j), kind = K == kBoxScene ? 1 : __ldg(S.pkind + i);
        const float e = __ldg(S.seg_m32 + j) * kScrUp + dh;
        const float d = scr_prim(S, kind, i, p[0], p[1], p[2]);
        if (!(fabsf(d) - eps - e > 0.f)) return 0.f;
        float b = scr_isotropic<K>(kind, d, e, eps);
        if (b >= t) continue;
        const float4 A = __ldg(S.p32 + 2 * i), B = __ldg(S.p32 + 2 * i + 1);
        const float c[3] = {A.x, A.y, A.z}, h[3] = {B.x, B.y, B.z};
        if (kind == 1) b = fmaxf(b, d > 0.f ? scr_box_entry(c, h, e, p, u, eps) : scr_box_exit(c, h, e, p, u, eps));
        else if (kind == 0) b = fmaxf(b, scr_sphere(A, d, e, p, u, eps));
        t = fminf(t, b);
    }
    return t;
}

// A packet's ray in FP32.
struct Ray32 {
    float p[3], u[3], iu[3];                 // iu: 1 / |u|
};

// seg_box64 of the box P (centre, half extents; FP32: c, h), with the quotients of the
// axes that FP32 shows to count.  The reference takes an axis' smaller and
// larger quotient, which are those of the plane behind and ahead (rounding
// is monotone): from inside, the bound is the first plane ahead; from
// outside, the last plane behind, if it certainly lies before the first one
// ahead and ahead of the packet.
static __device__ __noinline__ double seg_face64(const double *P, const Ray32 &r, const float *c, const float *h,
                                                 bool inside, double px, double py, double pz, double ux, double uy,
                                                 double uz, double e, float ef, float eps)
{
    const float inf = __int_as_float(0x7f800000);
    float lo[3], hi[3];                      // bounds of the distance of the face that counts
    float ahead = inf, behind = -inf, last = -inf;
    bool odd = false;                        // a direction component of zero, a box thinner than 2 e
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float g = inside ? h[a] - ef : h[a] + ef;
        const float q = r.u[a] > 0.f ? r.p[a] - c[a] : c[a] - r.p[a];
        odd = odd || r.u[a] == 0.f || !(g > eps);
        const float at = (inside ? g : -g) - q;
        const float x = (at - eps) * r.iu[a], y = (at + eps) * r.iu[a];
        lo[a] = x - 1e-5f * fabsf(x); hi[a] = y + 1e-5f * fabsf(y);
        ahead = fminf(ahead, inside ? hi[a] : (g - q - eps) * r.iu[a] * kScrDown);
        behind = fmaxf(behind, lo[a]);
        last = fmaxf(last, hi[a]);
    }
    // from outside: certainly hit (the last plane behind before the first ahead) and ahead
    if (eps == 0.f || odd || !(fabsf(ahead) < 1e30f) || (!inside && !(behind > 0.f && last < ahead)))
        return seg_box64(P[0], P[1], P[2], P[3], P[4], P[5], inside ? -1.0 : 1.0, px, py, pz, ux, uy, uz, e);
    double t = __longlong_as_double(inside ? 0x7ff0000000000000LL : (long long)0xfff0000000000000ULL);
#pragma unroll 1
    for (int a = 0; a < 3; ++a) {
        if (a == 0 ? (inside ? lo[0] > ahead : hi[0] < behind)
                   : a == 1 ? (inside ? lo[1] > ahead : hi[1] < behind) : (inside ? lo[2] > ahead : hi[2] < behind))
            continue;
        const double p = a == 0 ? px : a == 1 ? py : pz, u = a == 0 ? ux : a == 1 ? uy : uz;
        const double he = inside ? P[3 + a] - e : P[3 + a] + e;
        const bool plus = (__double2hiint(u) >= 0) == inside;
        const double x = div64((plus ? P[a] + he : P[a] - he) - p, u);
        t = inside ? min64(t, x) : max64(t, x);
    }
    return __double2hiint(t) >= 0 ? t : 0.0;
}

// An upper bound of the exit from a box certainly around p (else inf).
__device__ __forceinline__ float scr_exit_most(const Ray32 &r, const float *c, const float *h, float e, float eps)
{
    float t = __int_as_float(0x7f800000);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float q = r.u[a] > 0.f ? r.p[a] - c[a] : c[a] - r.p[a];
        if (!(fabsf(q) + e + eps < h[a])) return __int_as_float(0x7f800000);
        if (r.u[a] != 0.f) t = fminf(t, (h[a] - q + eps) * r.iu[a] * kScrUp);
    }
    return t;
}

// The move bound of segment_bound64, leaving out what cannot lower it: first
// an FP32 upper bound of the result (cap), then, in the reference's order, the
// surfaces that FP32 does not show to lie beyond it or beyond the smallest so
// far.  E and C: the evaluation at p and its screening, which know the nearest
// surface's distance and a fold's list.  A call took 26000 to 43000 cycles
// (layered slab, vessel tree), most of it for surfaces that did not count, for
// conversions of FP64 tables that FP32 copies exist of (64 cycles each, as any
// FP64 operation), and for the tree's fold a second time: vessel tree 1e4
// packets 33.9 -> 26.2 ms, 4e4 51.4 -> 39.0, layered slab 1e5 44.7 -> 42.5.
//
// The reference passes a surface over when |d| - e is not below its bound so
// far.  For all but a box seen from outside, whose ray bound may be smaller
// than |d| - e (scr_isotropic), that changes nothing.  Surfaces left out here
// lie beyond the bound so far, or beyond cap: then the reference's bound so
// far may be another one above cap, and a box with |d| - e between cap and
// ours may be one that it passes over.  Plain scenes start again without cap
// there.  In scenes of simple regions (e = delta / 2 for every box) the result
// cannot depend on it: cap exceeds the result by feps at least, and each such
// box can only bring the bounds in question down by 0.74 delta / 2, all of
// them together by less than feps has room for.
template <int K>
static __device__ __noinline__ double segment_bound64_screened(const DevScene &S, const Eval64 &E, const Screen64 &C,
                                                               double px, double py, double pz, double ux, double uy,
                                                               double uz)
{
    const float eps = S.feps;
    Ray32 r;
    r.p[0] = (float)px; r.p[1] = (float)py; r.p[2] = (float)pz;
    r.u[0] = (float)ux; r.u[1] = (float)uy; r.u[2] = (float)uz;
    for (int a = 0; a < 3; ++a) r.iu[a] = __fdividef(1.f, fabsf(r.u[a]));
    const float *const p = r.p, *const u = r.u;
    const double dh = 0.5 * S.delta;
    const float dhf = (float)dh;
    static_assert(offsetof(DevScene, bbh) == offsetof(DevScene, bbc) + 3 * sizeof(double), "centre, half extents");
    const double *box = reinterpret_cast<const double *>(reinterpret_cast<const char *>(&S) + offsetof(DevScene, bbc));
    float cap = __int_as_float(0x7f800000);
    if (eps > 0.f) {
        cap = scr_exit_most(r, S.bbc32, S.bbh32, dhf * kScrUp, eps);
        for (int j = 0; j < S.nseg; ++j) {
            const int i = __ldg(S.seg_prims + j);
            if (K != kBoxScene && __ldg(S.pkind + i) != 1) continue;
            const float4 A = __ldg(S.p32 + 2 * i), B = __ldg(S.p32 + 2 * i + 1);
            const float c[3] = {A.x, A.y, A.z}, h[3] = {B.x, B.y, B.z};
            cap = fminf(cap, scr_exit_most(r, c, h, __ldg(S.seg_m32 + j) * kScrUp + dhf * kScrUp, eps));
        }
        cap *= kScrUp;
    }
    for (;;) {
        bool again = false;
        double t = __longlong_as_double(0x7ff0000000000000LL);
        if (!(eps > 0.f && scr_box_exit(S.bbc32, S.bbh32, dhf * kScrUp, p, u, eps) > cap))
            t = seg_face64(box, r, S.bbc32, S.bbh32, true, px, py, pz, ux, uy, uz, dh, dhf, eps);
        if (!one_each<K>() && S.soft_mask != 0ull && !(C.soft - dhf * kScrUp > fminf(cap, (float)t * kScrUp))) {
            double ds = __longlong_as_double(0x7ff0000000000000LL);
            for (unsigned long long m = S.soft_mask; m != 0ull; m &= m - 1ull) {
                const int k = __ffsll((long long)m) - 1;
                double d = E.dmin;                   // the nearest surface's is known
                if (k != E.istar) {
                    unsigned long long list = C.list;
                    int cnt = C.cnt;
                    if (k != C.flr) fold_list<K>(S, k, px, py, pz, 0.f, list, cnt);
                    d = fabs(region_exact<K>(S, k, px, py, pz, list, cnt));
                }
                ds = min64(ds, d);
            }
            t = min64(t, ds - dh);
        }
        for (int j = 0; j < S.nseg; ++j) {
            const int i = __ldg(S.seg_prims + j);
            const int kind = K == kBoxScene ? 1 : __ldg(S.pkind + i);
            const double e = __ldg(S.seg_m64 + j) + dh;
            const float e32 = __ldg(S.seg_m32 + j) + dhf, ef = e32 * kScrUp, tu = fminf((float)t * kScrUp, cap);
            const float df = scr_prim(S, kind, i, p[0], p[1], p[2]);
            const float iso = fabsf(df) - eps - ef;
            const float4 A = __ldg(S.p32 + 2 * i), B = __ldg(S.p32 + 2 * i + 1);
            const float c[3] = {A.x, A.y, A.z}, h[3] = {B.x, B.y, B.z};
            if (eps > 0.f && iso > 0.f) {        // certainly outside the margin
                if (scr_isotropic<K>(kind, df, ef, eps) > tu) continue;
                if (kind == 1 &&
                    (df > 0.f ? scr_box_entry(c, h, ef, p, u, eps) : scr_box_exit(c, h, ef, p, u, eps)) > tu)
                    continue;
                if (kind == 0 && scr_sphere(A, df, ef, p, u, eps) > tu) continue;
            }
            // FP64 where FP32 leaves it open whether the primitive is passed over
            // (|d| within its margin, or |d| - e not below the bound so far)
            double d = (double)df;
            if (!(eps > 0.f && iso > 0.f && fabsf(df) + eps - ef * kScrDown * kScrDown < tu * kScrDown * kScrDown)) {
                d = prim64<false>(S, kind, i, px, py, pz);
                if (!(fabs(d) > e)) return 0.0;
                const double away = fabs(d) - e;
                if (away >= t) continue;
                if (K == kPlainScene && SMCRT_RARE(tu == cap && away >= (double)cap && t > (double)cap)) {
                    again = true;            // the reference's bound so far is not known
                    break;
                }
            }
            const double *P = S.p64 + 8 * i;
            double b;
            if (kind == 0)
                b = seg_sphere64(P, d, px, py, pz, ux, uy, uz, e);
            else if (kind == 1)
                b = seg_face64(P, r, c, h, !(d > 0.0), px, py, pz, ux, uy, uz, e, e32, eps);
            else
                b = seg_capsule64(P, d, px, py, pz, ux, uy, uz, e);
            t = min64(t, b);
        }
        if (K != kPlainScene || !again) return t;
        cap = __int_as_float(0x7f800000);
    }
}

// ---------------------------------------------------------------------------
// Track-length tally: tally64 with the grid clip left out where the segment
// starts inside the grid, and the voxel index taken from FP32 where its
// fraction is clear of a voxel face.  Positions are in voxels from the grid's
// corner; the error of one is below DevScene.gr32 = 16 u (R / dl + n), or gm32
// = 16 u n from an FP64 difference.  A segment inside one voxel (most of them)
// takes one FP64 operation.
//
// A longer one walks in fixed point.  What a voxel gets is the integer nearest
// to 2^32 w times a piece's length, so the pieces need no more digits than
// decide that: distances along the segment are 64-bit integers in units of
// 2^-tfix, at least 2^-58 of the scene's size, 26 bits below the tally's own
// unit.  They come from one approximate reciprocal per axis (5 FP64 operations
// per axis, all told) and are stepped by additions; the reference takes 12 FP64
// operations per crossing, a rounded quotient each.
//
// Error.  With p exact, the reference's quotient fl(fl(plane_k - p) / u), where
// plane_k = fl(lo + fl(k dl)), and the integer fl(plane_k0 - p) r + (k - k0)
// fl(dl r), |r u - 1| < 2^-51, differ by less than 2^-53 / |u| times 2 (hi - lo)
// + 2 max(|lo|, |hi|) (the rounded planes k0 and k) + (hi - lo) + dl (the
// differences), on the grid's last plane 2 (hi - lo) more (its own face clips
// the segment there): DevScene.tq, an axis' e; by 2^-50 t for r and the
// products; and by one unit per addition: slack.  Where an order of planes, a
// piece's sign or its rounding is closer than the errors, the FP64 walk goes on
// from the last plane.  Homogeneous sphere 3e4 packets (200^3 grid) 16.9 -> 9.0
// ms, glass sphere in a beam 3e5 16.8 -> 5.8 ms, vessel tree 1e4 35.2 -> 33.3
// ms, layered slab 1e6 332 -> 325 ms.
// ---------------------------------------------------------------------------
// The rest of a walk of a segment that starts inside the grid, in FP64 (clipped at the grid's far faces).
static __device__ __noinline__ unsigned walk_rest64(const DevScene &S, long long *flu, double px, double py, double pz,
                                                    double ux, double uy, double uz, int ix, int iy, int iz, double t,
                                                    double len, double w)
{
    double tin = 0.0, tout = len;
    clip64(S.g_lo[0], S.g_hi[0], px, ux, tin, tout);
    clip64(S.g_lo[1], S.g_hi[1], py, uy, tin, tout);
    clip64(S.g_lo[2], S.g_hi[2], pz, uz, tin, tout);
    return walk64(S, flu, px, py, pz, ux, uy, uz, ix, iy, iz, t, tout, w);
}

// A number >= 0 in units of 2^-e, rounded down; those from 2^64 units on: 2^62.
__device__ __forceinline__ unsigned long long fixed64(double x, int e)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned long long m = (b & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull;
    const int s = (int)(b >> 52) - 1075 + e;
    return s >= 0 ? s > 11 ? 1ull << 62 : m << s : s < -63 ? 0ull : m >> -s;
}

// The plane i of one axis.
__device__ __forceinline__ double grid_plane(const DevScene &S, int a, int i)
{
    return __ldg(S.planes + (a == 0 ? 0 : a == 1 ? S.g_n[0] + 1 : S.g_n[0] + S.g_n[1] + 2) + i);
}

// One axis of a fixed-point walk: the distance of the plane ahead along the
// segment, its step from plane to plane, and the error of any of them (see
// below).  far: the plane lies certainly beyond the end.  False: the error
// is too large (a direction almost along the planes).
struct FixAxis {
    long long t, dt, e;
};

__device__ __forceinline__ bool fix_axis(const DevScene &S, int a, int &i, double p, double u, bool far, FixAxis &o)
{
    o.t = 1ll << 62;
    o.dt = 0;
    o.e = 0;
    if (far || u == 0.0) return true;
    const float iu = __fdividef(1.f, fabsf((float)u)), e = S.tq[a] * iu * kScrUp;
    if (!(e < 1e9f) || !(iu > 0.5f)) return false;
    o.e = (long long)(int)e + 1;
    // 1 / |u| from the FP32 reciprocal (relative error f below 2^-21): f^3 is
    // beyond FP64
    const double ua = fabs(u);
    const double r0 = __longlong_as_double(((long long)__float_as_int(iu) << 29) + (896ll << 52));
    const double f = __fma_rn(-ua, r0, 1.0);
    const double r = __fma_rn(r0, __fma_rn(f, f, f), r0);
    const unsigned long long most = 1ull << 62;
    const bool up = __double2hiint(u) >= 0;
    const double way = grid_plane(S, a, i + up) - p;
    o.dt = (long long)min(most, fixed64(S.g_dl[a] * r, S.tfix));
    o.t = (long long)min(most, fixed64(fabs(way) * r, S.tfix));
    if ((__double_as_longlong(way) << 1) == 0) {     // on the plane: a crossing of no length
        i += up ? 1 : -1;
        o.t = o.dt;
    }
    return true;
}

static __device__ __noinline__ unsigned tally64_screened(const DevScene &S, long long *flu, double px, double py,
                                                         double pz, double ux, double uy, double uz, double len,
                                                         double w)
{
    if (!(len > 0.0) || !(w > 0.0)) return 0u;
    const float lf = (float)len;
    const int nx = S.g_n[0], ny = S.g_n[1], nz = S.g_n[2];
    const float ax = lf * (float)ux * S.g_idl32[0], ay = lf * (float)uy * S.g_idl32[1], az = lf * (float)uz * S.g_idl32[2];
    float mx = S.gr32[0], my = S.gr32[1], mz = S.gr32[2];
    float gx = ((float)px - S.g_lo32[0]) * S.g_idl32[0], gy = ((float)py - S.g_lo32[1]) * S.g_idl32[1],
          gz = ((float)pz - S.g_lo32[2]) * S.g_idl32[2];
    float bx = floorf(gx), by = floorf(gy), bz = floorf(gz);
    // starts inside the grid, clear of the voxel's faces?
    const auto within = [&]() {
        return gx > mx && gx < (float)nx - mx && gy > my && gy < (float)ny - my && gz > mz && gz < (float)nz - mz;
    };
    // both ends beyond one side of the grid: no voxel
    const auto outside = [&]() {
        const float hx = gx + ax, hy = gy + ay, hz = gz + az;
        const float ex = mx + 1e-6f * (fabsf(gx) + fabsf(ax)), ey = my + 1e-6f * (fabsf(gy) + fabsf(ay)),
                    ez = mz + 1e-6f * (fabsf(gz) + fabsf(az));
        return fminf(gx, hx) > (float)nx + ex || fmaxf(gx, hx) < -ex || fminf(gy, hy) > (float)ny + ey ||
               fmaxf(gy, hy) < -ey || fminf(gz, hz) > (float)nz + ez || fmaxf(gz, hz) < -ez;
    };
    const auto clear = [](float g, float b, float m) { return fminf(g - b, b + 1.f - g) > 2.f * m; };
    if (!(within() && clear(gx, bx, mx) && clear(gy, by, my) && clear(gz, bz, mz))) {
        if (outside()) return 0u;
        // FP64 differences, and the index itself where that is not enough
        mx = S.gm32[0]; my = S.gm32[1]; mz = S.gm32[2];
        const double ox = px - S.g_lo[0], oy = py - S.g_lo[1], oz = pz - S.g_lo[2];
        gx = (float)ox * S.g_idl32[0]; gy = (float)oy * S.g_idl32[1]; gz = (float)oz * S.g_idl32[2];
        if (outside()) return 0u;
        if (!within()) return tally64(S, flu, px, py, pz, ux, uy, uz, len, w);
        bx = floorf(gx); by = floorf(gy); bz = floorf(gz);
        if (!clear(gx, bx, mx)) bx = (float)floor(div64(ox, S.g_dl[0]));
        if (!clear(gy, by, my)) by = (float)floor(div64(oy, S.g_dl[1]));
        if (!clear(gz, bz, mz)) bz = (float)floor(div64(oz, S.g_dl[2]));
    }
    int ix = (int)bx, iy = (int)by, iz = (int)bz;
    float sx = gx - bx, sy = gy - by, sz = gz - bz;          // position in the voxel
    // voxels to the plane ahead of each axis, and 1 / (voxels the segment advances)
    // (a direction of zero has none)
    sx = ax > 0.f ? 1.f - sx : ux == 0.0 ? 1e6f : sx;
    sy = ay > 0.f ? 1.f - sy : uy == 0.0 ? 1e6f : sy;
    sz = az > 0.f ? 1.f - sz : uz == 0.0 ? 1e6f : sz;
    const float vx = __fdividef(1.f, fmaxf(fabsf(ax), 1e-30f)), vy = __fdividef(1.f, fmaxf(fabsf(ay), 1e-30f)),
                vz = __fdividef(1.f, fmaxf(fabsf(az), 1e-30f));
    // where the planes ahead certainly do not lie before, along the segment
    // (1 = its end)
    const float lx = (sx - 2.f * mx) * vx * kScrDown, ly = (sy - 2.f * my) * vy * kScrDown,
                lz = (sz - 2.f * mz) * vz * kScrDown;
    if (fminf(lx, fminf(ly, lz)) > kScrUp) {                 // all of it in this voxel
        red_add(flu + ((long long)iz * ny + iy) * nx + ix, fx64(w * len));
        return 1u;
    }
    // the walk in fixed point
    FixAxis X, Y, Z;
    bool ok = S.tfix != 0 && w <= 1.0;
    ok = ok && fix_axis(S, 0, ix, px, ux, lx > kScrUp, X);
    ok = ok && fix_axis(S, 1, iy, py, uy, ly > kScrUp, Y);
    ok = ok && fix_axis(S, 2, iz, pz, uz, lz > kScrUp, Z);
    if (!ok) return walk_rest64(S, flu, px, py, pz, ux, uy, uz, (int)bx, (int)by, (int)bz, 0.0, len, w);
    if ((unsigned)ix >= (unsigned)nx || (unsigned)iy >= (unsigned)ny || (unsigned)iz >= (unsigned)nz) return 0u;
    const int shift = S.tfix - 33;
    const unsigned long long half = 1ull << (shift - 1);
    const unsigned long long wf = fixed64(w, 63);
    const long long tl = (long long)min(1ull << 60, fixed64(len, S.tfix));
    long long slack = (tl >> 49) + 16;
    long long *at = flu + ((long long)iz * ny + iy) * nx + ix;
    const long long row = nx, sheet = (long long)nx * ny;
    long long t = 0, et = 0;
    int last = -1;                           // the axis of the plane at t
    unsigned npieces = 0u;
    for (;;) {
        const bool cx = X.t <= Y.t && X.t <= Z.t, cy = !cx && Y.t <= Z.t;
        const long long tn = cx ? X.t : cy ? Y.t : Z.t, en = (cx ? X.e : cy ? Y.e : Z.e) + slack;
        const long long o1 = cx ? Y.t - Y.e : X.t - X.e, o2 = cx || cy ? Z.t - Z.e : Y.t - Y.e;
        const long long other = min(o1, o2);
        const bool ends = min(tn - en, other) > tl + slack;
        const long long p = (ends ? tl : tn) - t, err = et + (ends ? 0 : en) + slack;
        const unsigned long long v = __umul64hi(wf, (unsigned long long)p) + half;
        const long long ev = (long long)__umul64hi(wf, (unsigned long long)err) + 16;
        const long long frac = (long long)(v & (2ull * half - 1ull));
        if (!((ends || (tn + en < other && tn + en < tl)) && p > err && frac > ev &&
              frac + ev < (long long)(2ull * half))) {
            // too close to call: FP64 from the plane at t on
            double te = 0.0;
            if (last >= 0) {
                const int i = last == 0 ? ix : last == 1 ? iy : iz;
                const double u = last == 0 ? ux : last == 1 ? uy : uz, q = last == 0 ? px : last == 1 ? py : pz;
                te = div64(grid_plane(S, last, u > 0.0 ? i : i + 1) - q, u);
            }
            return npieces + walk_rest64(S, flu, px, py, pz, ux, uy, uz, ix, iy, iz, te, len, w);
        }
        red_add(at, (long long)(v >> shift));
        npieces += 1u;
        if (ends) return npieces;
        t = tn;
        et = en;
        slack += 2;
        if (cx) {
            last = 0;
            X.t += X.dt;
            if (ux > 0.0 ? ++ix >= nx : --ix < 0) return npieces;
            at += ux > 0.0 ? 1 : -1;
        } else if (cy) {
            last = 1;
            Y.t += Y.dt;
            if (uy > 0.0 ? ++iy >= ny : --iy < 0) return npieces;
            at += uy > 0.0 ? row : -row;
        } else {
            last = 2;
            Z.t += Z.dt;
            if (uz > 0.0 ? ++iz >= nz : --iz < 0) return npieces;
            at += uz > 0.0 ? sheet : -sheet;
        }
    }
}

}  // namespace smcrt
