// smcrt_internal.h -- structures shared by the host runtime (smcrt_api.cpp)
// and the two packet-kernel translation units (FP64 and mixed precision).
// Not part of the public C-ABI.
#pragma once

#include <cmath>
#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/smcrt.h"

namespace smcrt {

constexpr int kMaxStack = 4;      // CSG register stack depth on the device
constexpr int kMaxRegions = 64;
constexpr int kMaxPrims = 4096;
constexpr int kMaxGridSide = 1024;
constexpr int kMaxThreads = 128;
// Longest region program (instructions) whose normal the mixed kernel takes
// from the analytic SDF gradient; longer programs use six shared probes.
constexpr int kAnalyticNormalMaxInstr = 4;
// Fold regions with at least this many primitives get a culling grid.
constexpr int kCullMinPrims = 16;
// Cells per axis of the culling grid.  Finer cells list fewer candidates (the
// reach R is one cell): on the 64-capsule vessel scene 32 cells per axis
// beat 16 by 11 % with segment stepping and 22 % with sphere tracing.
constexpr int kCullGrid = 32;

// Device primitive kind: the smcrt_prim_kind, plus this bit when the
// primitive is evaluated in its own frame (smcrt_xform).  Instr.op carries
// it in bits 8..15, the DevScene.pkind table as is.
constexpr int32_t kXformFlag = 0x10;
constexpr int kXf64 = 20;   // doubles per primitive frame: R (9), t (3), s, op, a (4), 2 unused
constexpr int kXf32 = 5;    // float4 per primitive frame: R^T rows | t, (s, 1/s, op, 0), a

inline int32_t device_kind(const smcrt_prim &P) { return P.kind | (P.xform > 0 ? kXformFlag : 0); }

// The tables of primitive i: FP64 (8 doubles), FP32 (2 float4), and, when
// xd / xf are given and the primitive has a frame, the frame (kXf64 doubles,
// kXf32 float4).  Doubles are the caller's values or the reference's
// expressions (capsule: b - a and |b - a|^2), so the FP64 kernel computes
// with the same numbers as the oracle.
inline void fill_prim(const smcrt_scene *sc, int i, double *d, float4 *f, double *xd, float4 *xf)
{
    const smcrt_prim &P = sc->prims[i];
    for (int k = 0; k < 8; ++k) d[k] = 0.0;
    f[0] = make_float4(0.f, 0.f, 0.f, 0.f);
    f[1] = f[0];
    if (P.kind == SMCRT_CAPSULE) {
        const double bax = P.p[3] - P.p[0], bay = P.p[4] - P.p[1], baz = P.p[5] - P.p[2];
        const double baba = bax * bax + bay * bay + baz * baz;
        d[0] = P.p[0]; d[1] = P.p[1]; d[2] = P.p[2];
        d[3] = bax; d[4] = bay; d[5] = baz; d[6] = P.p[6]; d[7] = baba;
        f[0] = make_float4((float)P.p[0], (float)P.p[1], (float)P.p[2], (float)P.p[6]);
        f[1] = make_float4((float)bax, (float)bay, (float)baz, (float)(1.0 / baba));
    } else if (P.kind == SMCRT_BOX) {
        for (int k = 0; k < 6; ++k) d[k] = P.p[k];
        f[0] = make_float4((float)P.p[0], (float)P.p[1], (float)P.p[2], 0.f);
        f[1] = make_float4((float)P.p[3], (float)P.p[4], (float)P.p[5], 0.f);
    } else if (P.kind == SMCRT_TORUS || P.kind == SMCRT_CYLINDER) {
        for (int k = 0; k < 5; ++k) d[k] = P.p[k];
        f[0] = make_float4((float)P.p[0], (float)P.p[1], (float)P.p[2], (float)P.p[3]);
        f[1] = make_float4((float)P.p[4], 0.f, 0.f, 0.f);
    } else {
        for (int k = 0; k < 4; ++k) d[k] = P.p[k];
        f[0] = make_float4((float)P.p[0], (float)P.p[1], (float)P.p[2], (float)P.p[3]);
    }
    if (xd == nullptr || xf == nullptr) return;
    for (int k = 0; k < kXf64; ++k) xd[k] = 0.0;
    for (int k = 0; k < kXf32; ++k) xf[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (P.xform <= 0) return;
    const smcrt_xform &X = sc->xforms[P.xform - 1];
    for (int k = 0; k < 9; ++k) xd[k] = X.rot[k];
    for (int k = 0; k < 3; ++k) xd[9 + k] = X.t[k];
    xd[12] = X.s;
    xd[13] = (double)X.op;
    for (int k = 0; k < 4; ++k) xd[14 + k] = X.a[k];
    const double *R = X.rot;
    xf[0] = make_float4((float)R[0], (float)R[3], (float)R[6], (float)X.t[0]);
    xf[1] = make_float4((float)R[1], (float)R[4], (float)R[7], (float)X.t[1]);
    xf[2] = make_float4((float)R[2], (float)R[5], (float)R[8], (float)X.t[2]);
    xf[3] = make_float4((float)X.s, (float)(1.0 / X.s), (float)X.op, 0.f);
    xf[4] = make_float4((float)X.a[0], (float)X.a[1], (float)X.a[2], (float)X.a[3]);
}

// Primitives the mixed kernel's analytic normal and the culling grid handle:
// sphere, box, capsule in scene coordinates.
inline bool plain_prim(const smcrt_prim &P) { return P.kind <= SMCRT_CAPSULE && P.xform <= 0; }

// Segment stepping bounds a region by rays to its primitives, widened by a
// margin of k/4 per smooth union (a smooth union lies at most k/4 below
// min, and min, max and subtraction move by at most their operands'
// change, so the region's surface lies where some primitive has |d| <= the
// sum).  A region with more smooth unions than kSegMaxSmooth ("soft") keeps
// the isotropic bound |d| - delta/2; the last instruction of its program
// carries kSoftRegionEnd in Instr.op.
constexpr int kSegMaxSmooth = 8;
constexpr int32_t kSoftRegionEnd = 0x10000;

inline bool region_is_soft(const smcrt_scene *sc, int r)
{
    const smcrt_region &R = sc->regions[r];
    int n = 0;
    for (int i = 0; i < R.node_count; ++i)
        if (sc->nodes[R.node_begin + i].op == SMCRT_OP_SMOOTH_UNION) ++n;
    return n > kSegMaxSmooth;
}

// Sum of k/4 over region r's smooth unions, in program order (0: hard CSG).
inline double region_margin(const smcrt_scene *sc, int r)
{
    const smcrt_region &R = sc->regions[r];
    double m = 0.0;
    for (int i = 0; i < R.node_count; ++i)
        if (sc->nodes[R.node_begin + i].op == SMCRT_OP_SMOOTH_UNION) m = m + 0.25 * sc->nodes[R.node_begin + i].k;
    return m;
}

// The primitives whose offset surfaces bound a segment-stepping move: the
// distinct primitives of the regions that are not soft, in first-use order,
// each with the largest margin of those regions that use it.  skip_region
// (the mixed kernel's culled region) is left out: its culled distance
// bounds moves isotropically (ray bounds over all its primitives would undo
// the culling).  Writes at most kMaxPrims entries; no allocation.
inline int seg_entries(const smcrt_scene *sc, int32_t *out, double *margin, int skip_region = -1)
{
    int16_t at[kMaxPrims];   // entry of a primitive + 1 (kMaxPrims fits)
    for (int i = 0; i < sc->nprims && i < kMaxPrims; ++i) at[i] = 0;
    int n = 0;
    for (int r = 0; r < sc->nregions; ++r) {
        if (r == skip_region || region_is_soft(sc, r)) continue;
        const smcrt_region &R = sc->regions[r];
        const double m = region_margin(sc, r);
        for (int i = 0; i < R.node_count; ++i) {
            const smcrt_csg_node &nd = sc->nodes[R.node_begin + i];
            if (nd.op != SMCRT_OP_PRIM || nd.prim < 0 || nd.prim >= sc->nprims || nd.prim >= kMaxPrims) continue;
            if (at[nd.prim] == 0) {
                margin[n] = 0.0;
                out[n] = nd.prim;
                at[nd.prim] = (int16_t)++n;
            }
            double &e = margin[at[nd.prim] - 1];
            e = std::fmax(e, m);
        }
    }
    return n;
}

// FP64 optics of a region: mu_a, mu_s, g, n, mu_t, albedo, and the constants of
// its scattering: 1 / mu_t, 1 - g g, 1 - g, 2 g, 1 + g g, 1 / (2 g).
constexpr int kReg64 = 12;

inline void fill_reg64(const smcrt_region &R, double *d)
{
    const double mu_t = R.mu_a + R.mu_s;
    d[0] = R.mu_a; d[1] = R.mu_s; d[2] = R.g; d[3] = R.n;
    d[4] = mu_t;
    d[5] = mu_t > 0.0 ? R.mu_s / mu_t : 0.0;
    d[6] = mu_t > 0.0 ? 1.0 / mu_t : 0.0;
    d[7] = 1.0 - R.g * R.g;
    d[8] = 1.0 - R.g;
    d[9] = 2.0 * R.g;
    d[10] = 1.0 + R.g * R.g;
    d[11] = R.g != 0.0 ? 1.0 / (2.0 * R.g) : 0.0;
}

// The grid's planes lo + i dl of the three axes in turn (nx + 1, ny + 1,
// nz + 1 of them).
inline size_t plane_count(const smcrt_grid *g) { return (size_t)g->n[0] + g->n[1] + g->n[2] + 3; }

inline void fill_planes(const smcrt_grid *g, double *d)
{
    for (int a = 0; a < 3; ++a) {
        const double dl = (g->hi[a] - g->lo[a]) / (double)g->n[a];
        for (int i = 0; i <= g->n[a]; ++i) *d++ = g->lo[a] + (double)i * dl;
    }
}

// Device instruction (compiled CSG program).  op: 0 push primitive;
// 1 union, 2 smooth union, 3 intersect, 4 subtract.  prim >= 0 with a
// binary op means "combine the stack top (left) with this primitive
// (right)"; prim < 0 with a binary op combines the top two stack entries.
// region >= 0 marks the last instruction of that region's program.
struct Instr {
    int32_t op;
    int32_t prim;
    int32_t region;
    int32_t pad;
};

// Scenes of simple regions (a compiled program): every region one box; one
// sphere, box or capsule; or one box or a left fold of unions and smooth
// unions of two or more capsules.  All in scene coordinates.
enum : int { kSinglePrims = 1, kSingleBoxes = 2, kSingleTree = 3 };
inline int single_regions(const Instr *ins, const int2 *rr, int nregions)
{
    bool one = true, box = true, tree = true;
    for (int r = 0; r < nregions; ++r) {
        const bool alone = rr[r].y - rr[r].x == 1;
        for (int i = rr[r].x; i < rr[r].y; ++i) {
            const int op = ins[i].op & 0xff, kind = (ins[i].op >> 8) & 0xff;
            one = one && alone && kind <= SMCRT_CAPSULE;
            box = box && alone && kind == SMCRT_BOX;
            tree = tree && ins[i].prim >= 0 &&
                   (alone ? kind == SMCRT_BOX
                          : kind == SMCRT_CAPSULE && (i == rr[r].x || op == SMCRT_OP_UNION || op == SMCRT_OP_SMOOTH_UNION));
        }
    }
    return box ? kSingleBoxes : one ? kSinglePrims : tree ? kSingleTree : 0;
}

// Scene + source + grid of one plan as the kernels read them.  Lives in
// device memory; each warp stages a copy in shared memory when it starts
// on a job.  All double fields are computed on the host with the same
// expressions the FP64 reference uses, so the FP64 kernel sees identical
// values.
struct DevScene {
    // instruction stream and primitive tables (device pointers)
    const Instr *instr;
    const double *k64;        // smooth radius per instruction
    const float *kinv32;      // 1/k per instruction (FP32 path)
    const int32_t *pkind;     // per primitive: 0 sphere, 1 box, 2 capsule
    const double *p64;        // 8 per primitive (capsule: a, b-a, r, |b-a|^2)
    const float4 *p32;        // 2 per primitive (capsule: a|r, b-a|1/|b-a|^2)
    const int2 *rrange;       // per region: instruction [begin, end)
    const double *reg64;      // kReg64 per region (fill_reg64)
    const float4 *reg32;      // per region: mu_t, albedo, g, n
    int32_t ninstr, nregions, nprims, precision;
    // bounding box as centre / half extent
    double bbc[3], bbh[3];
    float bbc32[3], bbh32[3];
    double delta, ambient_n;
    float delta32;            // FP32 surface threshold (>= 64 ulp of the scene extent)
    float ambient_n32;
    int32_t analytic_nrm;     // mixed mode: normals from the analytic SDF gradient (short programs)
    // Spatial culling of one long fold region (mixed mode only): a G^3 grid
    // of cells, each listing the region's primitives within distance R of
    // the cell; elsewhere the region's value is bounded by R - k/4.
    int32_t cull_region;      // -1: none
    int32_t cull_g;
    int32_t cull_op;          // 1 union, 2 smooth union
    int32_t cull_kind;        // kListCapsules: only capsules listed; kListTree: and every other region is one box
    float cull_lo[3], cull_inv_s[3];
    float cull_rmax;          // R (union) or R - k/4 (smooth union)
    float cull_kinv;
    const int32_t *cull_off;  // G^3 + 1 prefix offsets into cull_list
    const int32_t *cull_list; // primitive indices, in the region's fold order
    // Segment stepping (enum smcrt_stepping): the bounding primitives and
    // their margins (sum of k/4 over the smooth unions of their regions)
    const int32_t *seg_prims;
    const double *seg_m64;
    const float *seg_m32;
    int32_t stepping, nseg;
    // Primitive frames (kXf64 doubles / kXf32 float4 per primitive), null
    // when no primitive has one
    const double *xf64;
    const float4 *xf32;
    int32_t general;          // some primitive is a torus or cylinder or has a frame
    int32_t singles;          // single_regions
    float h32;                // FP32 central-difference step for normals
    int64_t max_steps;
    // source
    int32_t src_kind, pad0;
    double src_pos[3], src_dir[3], src_b1[3], src_b2[3], src_radius;
    float src_pos32[3], src_dir32[3], src_b132[3], src_b232[3], src_radius32;
    // grid (fluence voxels; n = 0 disables the tally)
    double g_lo[3], g_hi[3], g_dl[3];
    float g_lo32[3], g_hi32[3], g_dl32[3], g_idl32[3];
    int32_t g_n[3], pad1;
    // FP64 kernel: FP32 screening (smcrt_screen.cuh).  feps = 0: none.
    uint64_t screen_mask;     // regions whose FP32 value has an error below feps
    uint64_t fold_mask;       // regions that are left folds of unions and smooth unions
    uint64_t soft_mask;       // soft regions (segment stepping)
    float feps;               // error bound of an FP32 distance
    float gm32[3];            // error bound of an FP32 position in voxels from an FP64 difference, per axis
    float gr32[3];            // ... from FP32 coordinates
    float tq[3];              // fixed-point walk: error of a plane's distance times |u|, in units, per axis
    int32_t tfix;             // ... its unit is 2^-tfix (0: no fixed-point walk)
    int32_t matched;          // every region has the ambient index (default_variant)
    const double *planes;     // fill_planes (where tfix > 0)
};

// The range of the FP64 screening: every coordinate, half extent and radius
// of the scene and its source, plus four surface thresholds; 0 where there is
// no screening (general shapes, FP32 squares out of range).
inline double screen_range(const smcrt_scene *sc, const smcrt_source *src)
{
    double R = 0.0;
    const double spread = src->kind == SMCRT_SRC_DISC || src->kind == SMCRT_SRC_SQUARE ? src->radius : 0.0;
    for (int a = 0; a < 3; ++a) {
        R = std::fmax(R, std::fmax(std::fabs(sc->bbox_lo[a]), std::fabs(sc->bbox_hi[a])));
        R = std::fmax(R, std::fabs(src->pos[a]) + spread);
    }
    for (int i = 0; i < sc->nprims; ++i) {
        const smcrt_prim &P = sc->prims[i];
        if (!plain_prim(P)) return 0.0;
        for (int a = 0; a < 3; ++a) {
            if (P.kind == SMCRT_SPHERE) R = std::fmax(R, std::fabs(P.p[a]) + P.p[3]);
            else if (P.kind == SMCRT_BOX) R = std::fmax(R, std::fabs(P.p[a]) + P.p[3 + a]);
            else if (P.kind == SMCRT_CAPSULE)
                R = std::fmax(R, std::fmax(std::fabs(P.p[a]), std::fabs(P.p[3 + a])) + P.p[6]);
        }
    }
    R = R + 4.0 * sc->delta;
    return R > 1e-6 && R < 1e12 ? R : 0.0;
}

// The fixed-point walk's unit is 2^-walk_bits of a centimetre; 0: no such walk.
inline int walk_bits(double R)
{
    int k;
    std::frexp(R, &k);                           // R < 2^k: a move is shorter than 4 R <= 2^(k + 2)
    return R > 0.0 && 58 - k >= 40 ? 58 - k : 0;
}

// The screening fields of a compiled scene: the error bounds and region
// classes that smcrt_screen.cuh states.
inline void fill_screen(DevScene &H, const smcrt_scene *sc, const smcrt_source *src, const smcrt_grid *g,
                        const Instr *ins, const int2 *rr)
{
    const double R = screen_range(sc, src);
    H.screen_mask = H.fold_mask = H.soft_mask = 0;
    for (int r = 0; r < sc->nregions; ++r)       // bounds the moves, screened or not
        if (region_is_soft(sc, r)) H.soft_mask |= 1ull << r;
    H.feps = 0.f;
    H.tfix = 0;
    for (int a = 0; a < 3; ++a) H.gm32[a] = H.gr32[a] = INFINITY;
    if (R == 0.0) return;
    // the FP32 error; in scenes of simple regions also what the corners of all
    // boxes grown by delta / 2 could take from a bound (segment_bound64_screened)
    int nbox = 0;
    for (int i = 0; i < sc->nprims; ++i) nbox += sc->prims[i].kind == SMCRT_BOX;
    H.feps = (float)(R / 65536.0 + (H.singles ? 0.75 * (nbox + 1) * (0.5 * sc->delta) : 0.0));
    for (int r = 0; r < sc->nregions; ++r) {
        const uint64_t bit = 1ull << r;
        bool fold = rr[r].y - rr[r].x <= 60000;   // list entries are 16 bits
        int smooth = 0;
        for (int i = rr[r].x; i < rr[r].y; ++i) {
            const int op = ins[i].op & 0xff;
            if (op == SMCRT_OP_SMOOTH_UNION) ++smooth;
            if (i > rr[r].x && (ins[i].prim < 0 || (op != SMCRT_OP_UNION && op != SMCRT_OP_SMOOTH_UNION))) fold = false;
        }
        if (fold) H.fold_mask |= bit;
        if (fold || smooth <= 8) H.screen_mask |= bit;
    }
    H.tfix = walk_bits(R);
    for (int a = 0; a < 3; ++a) {
        const double Rg = std::fmax(R, std::fmax(std::fabs(g->lo[a]), std::fabs(g->hi[a])));
        const double dl = (g->hi[a] - g->lo[a]) / (double)g->n[a];
        const double span = g->hi[a] - g->lo[a], far = std::fmax(std::fabs(g->lo[a]), std::fabs(g->hi[a]));
        H.tq[a] = (float)std::ldexp(6.1 * span + 2.1 * far, H.tfix - 53);
        H.gm32[a] = (float)(g->n[a] * (16.0 / 16777216.0));
        H.gr32[a] = (float)((Rg / dl + (double)g->n[a]) * (16.0 / 16777216.0));
    }
}

// A packet parked between serving rounds: its complete state at a trace
// boundary (FP32 values are stored widened, which round-trips exactly), so
// resuming it later continues the same arithmetic and the same random stream.
struct DeferState {
    double p[3], u[3], w, tau;
    long long pA, pG;
    uint32_t id_lo, id_hi, event, nsteps, pscat, pad[3];
};

// Per-job deferral lists, double-buffered by round parity: a round resumes
// the packets parked in list `in` and parks its own stragglers in 1 - in.
struct JobDefer {
    unsigned count[2];
    unsigned cursor[2];
    DeferState *buf[2];
    unsigned cap;
    unsigned overflow;       // stragglers that found the list full (kept running)
};

// Work descriptor of one job in a launch.  `next` is the packet-id cursor
// the warps claim from with atomicAdd.
struct JobWork {
    unsigned long long next;      // next packet id to hand out
    unsigned long long end;       // one past the last id
    unsigned long long begin;     // first id (records are indexed id - begin)
    unsigned long long seed;
    long long *fluence;           // device, may be null
    smcrt_totals *totals;         // device
    smcrt_packet_record *records; // device, may be null
    const DevScene *scene;        // device
    int32_t cancelled;            // host-set: stop handing out ids
    int32_t defer_in;             // list resumed in this launch (0 / 1)
    JobDefer *defer;              // device, may be null (no parking)
    long long park_cycles;        // > 0: park a packet after this many SM cycles in the launch
    long long drain_cycles;       // > 0 (served rounds): once its warp finds no job with work left,
                                  // park a packet after this many SM cycles in the launch
    int32_t stage;                // mixed kernel: stage the scene tables in shared memory
    int32_t lanes;                // plan launches: lanes of a warp that carry packets (0 = all 32)
    int32_t *jstat;               // device, may be null: this job's own status word (bits OR-ed in)
    unsigned long long time_limit_ns;   // > 0: a warp stops this job that long after it started on it
};

// Kernel status word bits.
constexpr int kStatusBadJob = SMCRT_STATUS_BAD_JOB;
constexpr int kStatusStackOverflow = 2;
constexpr int kStatusTimeout = SMCRT_STATUS_TIMEOUT;

// Launch wrappers, one per translation unit; `variant` selects the register
// budget of the kernel instantiation (0 .. kNumVariants-1).
constexpr int kNumVariants = 3;
cudaError_t launch_fp64(JobWork *jobs, int njobs, int *status, int blocks, int threads,
                        cudaStream_t stream, int variant = 0);
cudaError_t launch_mixed(JobWork *jobs, int njobs, int *status, int blocks, int threads,
                         cudaStream_t stream, int variant = 0);
int occupancy_fp64(int threads, int variant = 0);
// Served rounds' FP64 kernel (3 blocks of 128 threads per SM).
cudaError_t launch_fp64_served(JobWork *jobs, int njobs, int *status, int blocks, int threads, cudaStream_t stream,
                               bool general);
int occupancy_fp64_served(int threads);
int occupancy_mixed(int threads, int variant = 0);
// Served rounds' mixed kernel, whose warps hold two jobs at a time (lanes
// refill from the next job instead of draining each): variant 0 / 1 = 5 / 4
// resident blocks of 128 threads, + kNumVariants * served_family.
cudaError_t launch_mixed_multi(JobWork *jobs, int njobs, int *status, int blocks, int threads,
                               cudaStream_t stream, int variant = 0);
int occupancy_mixed_multi(int threads, int variant = 0);
// FP64 plan launches of fewer packets than this run, unless the caller or the
// autotuner chose a shape, one block of 128 threads per SM with the largest
// register budget (variant 2): one warp per scheduler nearly fills the FP64
// pipe, and four warps disturb one another's instruction fetch less than
// twelve.  Measured, 1 x 128 against the 3 x 128 that larger launches run:
// layered slab 1e4 packets 13.5 / 17.4 ms, 1e5 41.5 / 44.3; vessel tree 1e4
// 26.8 / 35.5, 4e4 38.8 / 55.5; glass container 1e4 36.8 / 43.0, 1e5 74.5 /
// 79.5; shape gallery (general) 1e3 86.9 / 91.5, 1e4 191 / 221, 1e5 559 / 629,
// with sphere tracing 849 / 891.  Packets of short, even lives are better off
// with the wider launch well below the limit: sphere 1e4 3.5 / 4.6 ms, 1e5 10.9
// / 10.5, 5e5 47 / 40, with sphere tracing 163 / 146; layered slab 4e5 137 /
// 131, with sphere tracing 206 / 168; glass sphere in a beam 3e5 6.0 / 4.2;
// homogeneous sphere 1e5 19.2 / 16.1.
constexpr uint64_t kFewFp64Packets = 1u << 19;
constexpr int kFewFp64Variant = 2;

// Mixed plan launches run 4 blocks of 128 threads per SM with 128 registers
// (variant 1) unless the caller or the autotuner chose a shape, and 5 blocks
// with 96 registers (variant 0) from this many packets on in scenes without
// a cell list.  General scenes run 3 blocks (variant 2): their code exceeds the
// instruction cache (9.6 cycles of fetch stall per instruction with four
// blocks, 6.6 with three), and fewer warps disturb one another's fetch less.
// Measured, variant 0 / 1: layered slab 1e5 packets 3.22 / 3.03 ms, 5e5 7.36 / 7.83, 1e6 12.9 / 14.0, 1e7 111 / 124;
// with sphere tracing 4e5 15.0 / 14.7, 1e6 25.3 / 25.6; glass container 5e5
// 15.4 / 15.0, 1e6 21.4 / 21.6; thick slab 1e5 27.3 / 24.2, 4e5 37.6 / 35.3,
// 1e6 65.7 / 66.5; vessel tree 1e5 21.1 / 19.7, 4e6 98 / 96 ms; shape gallery,
// variants 0 / 1 / 2, 3e4 18.2 / 18.3 / 17.2, 1e5 53.2 / 53.7 / 49.1, 5e5 84.7 /
// 87.3 / 81.5, with sphere tracing 316 / 312 / 300.  (Layered slabs alone would
// cross over at 2e5; thick ones and sphere tracing near 1e6.)
//
// Scenes without an index step, whose packets meet no Fresnel surface, cross
// over earlier: homogeneous sphere (isotropic, optical radius 10) 6e4 packets
// 2.80 / 2.66 ms, 1e5 2.88 / 3.04, 6e5 8.80 / 10.16.
constexpr uint64_t kManyMixedPackets = 3u << 18;
constexpr uint64_t kManyMatchedPackets = 5u << 14;
inline bool matched_regions(const smcrt_scene *sc)
{
    bool all = true;
    for (int r = 0; r < sc->nregions; ++r) all = all && sc->regions[r].n == sc->ambient_n;
    return all;
}

// Variant of a plan launch whose shape nobody chose.
inline int default_variant(int precision, uint64_t npackets, const DevScene &S)
{
    if (precision == SMCRT_FP64) return npackets < kFewFp64Packets ? kFewFp64Variant : 1;
    if (S.general) return 2;
    return npackets < (S.matched ? kManyMatchedPackets : kManyMixedPackets) || S.cull_region >= 0 ? 1 : 0;
}

// Kernel family of a scene: its register variants start at kNumVariants
// times this.  The packet loop is close to the instruction cache's size, so
// code that a scene does not use costs it time all the same; a family's
// kernels leave out what its scenes cannot need:
//   general        tori, cylinders, frames, long programs (mixed: probe normals)
//   cell lists     mixed only; with general shapes or without
//   tree           a fold of capsules (mixed: a cell list) among regions of one
//                  box each
//   boxes          every region one box: no other shape, no CSG interpreter
//   singles        FP64: every region one sphere, box or capsule
//   plain          the rest: spheres, boxes and capsules, any CSG
// Measured, without and with the family.  Cell lists in the plain kernel / in
// their own: layered slab 1e7 packets 138.2 / 134.4 ms, 1e6 with sphere
// tracing 30.8 / 28.7, glass container 4e6 59.9 / 58.4; out of the general
// one: shape gallery 5e5 157 / 147 ms.  Tree: vessel tree 4e6 116 / 96 ms, 1e4
// 6.4 / 5.8; FP64 1e4 53.1 / 36.2, 4e4 80.4 / 56.5.  Boxes: layered slab 1e7 134.4 / 111.0 ms, 1e4 2.05 / 1.77, with
// sphere tracing 1e6 28.8 / 25.1, thick slab 1e6 67.7 / 65.3 (its loop is
// mostly scattering); FP64 layered slab 1e5 58.9 / 46.2 ms, 1e4 16.4 / 13.4,
// 1e6 485 / 342, thick slab 3e3 114.6 / 110.9.  Singles: FP64 sphere 1e5, with
// sphere tracing, 73.7 / 64.0 ms, segments 13.1 / 11.2; in mixed precision
// nothing (homogeneous sphere 2e6 24.8 / 25.2).  Served rounds hold scenes of
// several kinds and have three families (served_family).
enum : int { kPlainScene = 0, kGeneralScene = 1, kCulledScene = 2, kBoxScene = 3, kSingleScene = 4,
             kGeneralCulledScene = 5, kTreeScene = 6 };
enum : int { kListCapsules = 1, kListTree = 2 };   // DevScene.cull_kind
inline int scene_family(int precision, const DevScene &S)
{
    const bool cells = precision == SMCRT_MIXED && S.cull_region >= 0;
    if (S.general) return cells ? kGeneralCulledScene : kGeneralScene;
    if (cells) return S.cull_kind == kListTree ? kTreeScene : kCulledScene;
    if (S.singles == kSingleBoxes) return kBoxScene;
    if (precision == SMCRT_MIXED) return kPlainScene;
    return S.singles == kSinglePrims ? kSingleScene : S.singles == kSingleTree ? kTreeScene : kPlainScene;
}

// Families of the served rounds' kernels, of which a round takes the one that
// runs all its scenes: plain, plain with cell lists, general with cell lists.
inline int served_family(bool general, bool cells)
{
    return general ? kGeneralScene : cells ? kCulledScene : kPlainScene;
}

// Lanes of a warp that carry packets in a plan launch (JobWork.lanes; 0 =
// all).  A launch with fewer packets than lanes is bound by the latency of
// one loop iteration, which grows with the number of different branches a
// warp's lanes take, so its packets are spread evenly over all warps instead
// of filling the first ones.  Measured (layered slab, mixed, 3040 warps):
// 1e3 packets 1.61 ms with 1 lane against 2.61 ms with 32, 1e4 2.49 ms (4)
// against 3.32, 3e4 2.95 ms (6-8) against 3.70, 6e4 3.72 ms (16) against
// 3.91; FP64 (1824 warps): 1e3 18.1 ms (1) against 28.3, 1e4 43.3 ms (6)
// against 62.6.  Fewer lanes than this rule's serialise the packets.
inline int32_t spread_lanes(uint64_t npackets, int blocks, int threads)
{
    const uint64_t warps = (uint64_t)blocks * (uint64_t)(threads / 32);
    const uint64_t lanes = warps > 0 ? (npackets + warps - 1) / warps : 0;
    return lanes < 32 ? (int32_t)lanes : 0;
}
cudaError_t launch_set_job(JobWork *dst, const JobWork &v, cudaStream_t stream);
// Field validation of scene / source / grid, without compiling or
// allocating (host runtime).
int validate_scene(const smcrt_scene *sc, const smcrt_source *src, const smcrt_grid *g);

// Round prologue: for each table entry with a deferral list, zero the
// resume cursor of its input list and the count of its output list.
cudaError_t launch_round_prologue(JobWork *jobs, int njobs, cudaStream_t stream);

}  // namespace smcrt
