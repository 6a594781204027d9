// smcrt_k64.cu -- plain FP64 packet kernel (compiled with -fmad=false).
//
// Every floating-point step is an IEEE double operation in the order of the
// reference algorithm (Sec. 2.3 sphere tracing and interface handling,
// Eq. 1 free path, Sec. 3.1 HG scattering), so the int64 tallies equal the
// FP64 CPU reference bit for bit for any packet count.
#include "smcrt_screen.cuh"

namespace smcrt {

namespace {

// a / b given y = 1 / b rounded to nearest: two corrections of a y, each
// with the remainder from a fused multiply-add.  The result is the quotient
// rounded to nearest if its remainder is below half an ulp of it times b,
// which is compared exactly; otherwise (and near the range's ends) divides.
__device__ __forceinline__ double div_by64(double a, double b, double y)
{
    const double q0 = a * y;
    const double q = __fma_rn(__fma_rn(-b, q0, a), y, q0);
    const double r = __fma_rn(-b, q, a);
    const long long qb = __double_as_longlong(q) & 0x7fffffffffffffffLL, bb = __double_as_longlong(b) & 0x7fffffffffffffffLL;
    const int eq = (int)(qb >> 52), eb = (int)(bb >> 52);
    const long long half = bb + ((long long)(eq - 1076) << 52);
    const bool ok = eq > 700 && eq < 1400 && eb > 700 && eb < 1400 && (qb & 0x000FFFFFFFFFFFFFLL) != 0 &&
                    (__double_as_longlong(r) & 0x7fffffffffffffffLL) < half;
    return ok ? q : div64(a, b);
}

__device__ __forceinline__ double hg_cos64(const double *RG, double xi)
{   // Henyey-Greenstein inverse CDF (Sec. 3.1); isotropic for |g| < 1e-6
    const double g = __ldg(RG + 2);
    double c;
    if (fabs(g) < 1e-6) {
        c = 2.0 * xi - 1.0;
    } else {
        const double t = div64(__ldg(RG + 7), __ldg(RG + 8) + __ldg(RG + 9) * xi);
        c = div_by64(__ldg(RG + 10) - t * t, __ldg(RG + 9), __ldg(RG + 11));
    }
    return min64(max64(c, -1.0), 1.0);
}

// x / l for l = 1 + e, |e| < 2^-20: x - x e is the quotient but for a
// relative 2^-40, and its remainder tells exactly whether it is the one
// rounded to nearest (as in div_by64).
__device__ __forceinline__ double unit_div64(double x, double l, double e)
{
    const double q = __fma_rn(-x, e, x);
    const double r = __fma_rn(-l, q, x);
    const long long qb = __double_as_longlong(q) & 0x7fffffffffffffffLL;
    const int eq = (int)(qb >> 52);
    const long long half = __double_as_longlong(l) + ((long long)(eq - 1076) << 52);
    const bool ok = eq > 700 && (qb & 0x000FFFFFFFFFFFFFLL) != 0 &&
                    (__double_as_longlong(r) & 0x7fffffffffffffffLL) < half;
    return ok ? q : div64(x, l);
}

// x, y, z over their norm.  Directions are unit vectors up to rounding, so
// the square s of the norm is 1 + f with a tiny f.  For |f| < 2^-27 the root
// is 1 + f / 2 - f f / 8 + ..., below h = 1 + f / 2 by less than 2^-57; h is
// a floating-point number or lies halfway between two, so the root rounded
// to nearest is h rounded down: one fused multiply-add.  14 FP64 operations
// in place of 41.
__device__ __forceinline__ void normalise64(double &x, double &y, double &z)
{
    const double s = x * x + y * y + z * z;
    const int hs = __double2hiint(s);
    double l;
    if (hs >= 0x3fefffff && hs <= 0x3ff00000 && (hs == 0x3ff00000 ? (unsigned)__double2loint(s) < (1u << 25)
                                                                     : (unsigned)__double2loint(s) > 0xfc000000u))
        l = __fma_rd(s - 1.0, 0.5, 1.0);
    else
        l = sqrt64(s);
    const double e = l - 1.0;
    if ((__double2hiint(e) & 0x7fffffff) < 0x3eb00000) {   // |e| < 2^-20
        x = unit_div64(x, l, e);
        y = unit_div64(y, l, e);
        z = unit_div64(z, l, e);
    } else {
        x = div64(x, l);
        y = div64(y, l);
        z = div64(z, l);
    }
}

__device__ __forceinline__ double flip64(double x, double s)   // x times the sign of s
{
    return __longlong_as_double(__double_as_longlong(x) ^ (__double_as_longlong(s) & (long long)0x8000000000000000ULL));
}

// Rotation by the scattering angle; the azimuth from a Philox word.  The
// basis is onb64's, its products with the sign of uz (+-1) as sign flips.
__device__ __forceinline__ void scatter64(double &ux, double &uy, double &uz, double ct, uint32_t wphi)
{
    const double st = sqrt64((1.0 - ct) * (1.0 + ct));
    double sp, cp;
    sincos2pi_word(wphi, &sp, &cp);
    const double a = div64(-1.0, copysign(1.0, uz) + uz);
    const double b = ux * uy * a;
    const double sx = flip64(ux, uz);
    const double b1x = 1.0 + sx * ux * a, b1y = flip64(b, uz), b1z = -sx;
    const double b2y = copysign(1.0, uz) + uy * uy * a, b2z = -uy;
    const double a1 = st * cp, a2 = st * sp;
    double vx = a1 * b1x + a2 * b + ct * ux;
    double vy = a1 * b1y + a2 * b2y + ct * uy;
    double vz = a1 * b1z + a2 * b2z + ct * uz;
    normalise64(vx, vy, vz);
    ux = vx; uy = vy; uz = vz;
}

// Photon release (Sec. 2.1), out of line: position and direction from the
// source and the first optical depth (Eq. 1), from one Philox call's words.
struct Launched64 {
    double px, py, pz, ux, uy, uz, tau;
};

static __device__ __noinline__ Launched64 launch64(const DevScene &S, uint4 r)
{
    Launched64 o;
    const double x0 = u01_64(r.x), x3 = u01_64(r.w);
    o.px = S.src_pos[0]; o.py = S.src_pos[1]; o.pz = S.src_pos[2];
    o.ux = S.src_dir[0]; o.uy = S.src_dir[1]; o.uz = S.src_dir[2];
    if (S.src_kind == 1 || S.src_kind == 2) {
        double c1, c2;
        if (S.src_kind == 1) {
            const double rho = S.src_radius * sqrt64(x0);
            double sn, cs;
            sincos2pi_word(r.y, &sn, &cs);
            c1 = rho * cs;
            c2 = rho * sn;
        } else {
            c1 = S.src_radius * (2.0 * x0 - 1.0);
            c2 = S.src_radius * (2.0 * u01_64(r.y) - 1.0);
        }
        o.px = S.src_pos[0] + c1 * S.src_b1[0] + c2 * S.src_b2[0];
        o.py = S.src_pos[1] + c1 * S.src_b1[1] + c2 * S.src_b2[1];
        o.pz = S.src_pos[2] + c1 * S.src_b1[2] + c2 * S.src_b2[2];
    } else if (S.src_kind == 3) {
        const double ctt = 2.0 * x0 - 1.0;
        const double st = sqrt64((1.0 - ctt) * (1.0 + ctt));
        double sn, cs;
        sincos2pi_word(r.y, &sn, &cs);
        o.ux = st * cs; o.uy = st * sn; o.uz = ctt;
    }
    o.tau = -ln64(x3);
    return o;
}

// After a Fresnel decision at the surface point q (Sec. 2.3), out of line:
// the reflected or refracted direction and the point 2 delta beyond q on the
// packet's side (ee = 2 delta, signed like u.n).
struct Crossed64 {
    double px, py, pz, ux, uy, uz;
};

static __device__ __noinline__ Crossed64 cross64(double ux, double uy, double uz, double qx, double qy, double qz,
                                                 double nx, double ny, double nz, double cdot, double ee, double n1,
                                                 double n2, double ct, bool reflect)
{
    Crossed64 o;
    double sx;
    if (reflect) {
        const double c2 = 2.0 * cdot;
        ux = ux - c2 * nx; uy = uy - c2 * ny; uz = uz - c2 * nz;
        sx = -ee;
    } else {
        const double eta = div64(n1, n2);
        const double ci = fabs(cdot);
        const double k = (cdot > 0.0 ? 1.0 : -1.0) * (eta * ci - ct);
        ux = eta * ux - k * nx; uy = eta * uy - k * ny; uz = eta * uz - k * nz;
        sx = ee;
    }
    normalise64(ux, uy, uz);
    o.ux = ux; o.uy = uy; o.uz = uz;
    o.px = qx + sx * nx; o.py = qy + sx * ny; o.pz = qz + sx * nz;
    return o;
}

// Waiting packets are served when the lane iterations that they have waited
// reach the live lanes / kWaitExact (distances, about 100 FP64 operations)
// or / kWaitArrive (interfaces, about 250), against about 165 for an
// interaction.  Layered slab 1e5 packets: 60.9 ms with 3 and 2, 59.1 with 1
// for interfaces, 64.0 with 4; distances at once 62.7.
constexpr int kWaitExact = 3, kWaitArrive = 1;

struct WarpShared {
    DevScene S;
    WarpAcc acc;
    JobConst jc;
};

// Same iteration structure as the mixed kernel (refill, one scene
// evaluation, classify, one tally site, one Philox call, consumers), with
// every floating-point operation the reference algorithm's, in its order:
// the oracle's run of a packet is a sequence of the same IEEE operations on
// the same values, so its tallies come out bit for bit.
template <int K, bool SERVED>
__device__ bool run_job_fp64(const DevScene &S, WarpAcc *wa, const volatile JobConst *jc, JobWork *J,
                             int lane)
{
    const double delta = S.delta;

    // a small plan launch spreads its packets over all warps
    bool alive = false, retired = J->lanes > 0 && lane >= J->lanes;
    double px = 0, py = 0, pz = 0, ux = 0, uy = 0, uz = 0, w = 0, tau = 0;
    double dstar = 0;
    int phase = kTrace, istar = -1, reg = -1;
    int nsteps = 0;
    unsigned pscat = 0, npieces = 0, nev = 0;
    // lane iterations that packets have waited for FP64 distances and at
    // surfaces (warp-uniform), and a waiting packet's screening
    int wait_x = 0, wait_i = 0;
    unsigned long long kneg = 0ull, kmask = 0ull, klist = 0ull;
    float ksoft = 0.f, kdb = 0.f;
    int kfold = 0;
    long long pA = 0, pG = 0;
    uint32_t id_lo = 0, id_hi = 0, event = 0;
    uint32_t t_acq = 0;
    bool timed_out = false;              // the launch's time limit stopped the refills

    for (;;) {
        // ---- 1. refill: this job's parked packets first, then new ids
        {
            unsigned need = __ballot_sync(SMCRT_FULL, !alive && !retired);
            JobDefer *const dfr = (JobDefer *)jc->dfr;
            const int din = jc->din;
            if (SERVED && need && dfr != nullptr) {
                const int leader = __ffs(need) - 1;
                unsigned base = 0u, avail = 0u;
                if (lane == leader) {
                    // the counter also counts packets that found the list full
                    // (they kept running): only the first `cap` entries exist
                    avail = min(*(volatile unsigned *)&dfr->count[din], dfr->cap);
                    base = atomicAdd(&dfr->cursor[din], (unsigned)__popc(need));
                }
                base = __shfl_sync(SMCRT_FULL, base, leader);
                avail = __shfl_sync(SMCRT_FULL, avail, leader);
                if (!alive && !retired) {
                    const unsigned k = base + (unsigned)__popc(need & ((1u << lane) - 1u));
                    if (k < avail) {
                        const DeferState &d = dfr->buf[din][k];
                        px = (double)d.p[0]; py = (double)d.p[1]; pz = (double)d.p[2];
                        ux = (double)d.u[0]; uy = (double)d.u[1]; uz = (double)d.u[2];
                        w = (double)d.w; tau = (double)d.tau;
                        pA = d.pA; pG = d.pG;
                        id_lo = d.id_lo; id_hi = d.id_hi; event = d.event;
                        nsteps = (int)d.nsteps; pscat = d.pscat;
                        phase = kTrace;
                        t_acq = (uint32_t)clock();
                        alive = true;
                    }
                }
                need = __ballot_sync(SMCRT_FULL, !alive && !retired);
            }
            const bool want = !alive && !retired;
            if (need) {
                const int leader = __ffs(need) - 1;
                unsigned long long base = 0;
                if (lane == leader) {
                    if (*(volatile int32_t *)&J->cancelled) base = ~0ull;
                    else if (SMCRT_RARE(past_deadline(jc))) base = ~0ull - 1u;   // device time limit
                    else base = atomicAdd(&J->next, (unsigned long long)__popc(need));
                }
                base = __shfl_sync(SMCRT_FULL, base, leader);
                timed_out = timed_out || base == ~0ull - 1u;
                if (want) {
                    const unsigned long long id = base + (unsigned long long)__popc(need & ((1u << lane) - 1u));
                    if (base >= ~0ull - 1u || id >= jc->end) {
                        retired = true;
                    } else {
                        id_lo = (uint32_t)id;
                        id_hi = (uint32_t)(id >> 32);
                        event = 0u;
                        phase = kLaunch;
                        t_acq = (uint32_t)clock();
                        alive = true;
                    }
                }
            }
            if (__all_sync(SMCRT_FULL, retired)) break;
        }

        // ---- 2. the scene in FP32: where that shows that the packet
        // interacts before it can reach anything, no FP64 distance is needed
        Screen64 C;
        bool interact = false;
        const bool evals = alive && phase == kTrace;
        if (K == kGeneralScene) {
            if (evals) phase = kExact;
        } else if (evals) {
            C = scene_screen<K>(S, (float)px, (float)py, (float)pz, kForTrace);
            kneg = C.neg; kmask = C.mask; klist = C.list; kfold = C.flr << 8 | (C.cnt & 0xff);
            ksoft = C.soft; kdb = C.db;
            phase = kExact;
            if (C.lo > (float)delta * kScrUp) {          // clear of every surface, region known
                reg = C.neg != 0ull ? 63 - __clzll((long long)C.neg) : -1;
                const float m = reg >= 0 ? (float)__ldg(S.reg64 + kReg64 * reg + 4) : 0.f;
                const float need = (float)tau * (kScrUp * kScrUp);
                interact = m > 0.f && need < m * (C.lo - (float)delta);
                if (!interact && S.stepping == SMCRT_STEP_SEGMENT) {
                    const float p[3] = {(float)px, (float)py, (float)pz}, u[3] = {(float)ux, (float)uy, (float)uz};
                    interact = m > 0.f && need < m * segment_screen<K>(S, C.soft, p, u);
                }
            }
        }
        nev += evals;

        // ---- 3. FP64: the packets for which FP32 did not do, once enough of
        // them wait (an FP64 operation costs the same for one lane as for
        // all); moves, arrivals at a surface, escapes
        bool move = interact, fresnel = false, iter_done = false;
        bool fin = false;                      // the packet ends this iteration
        bool out = false;                      // ... leaving the volume: R or T
        long long fin_R = 0, fin_T = 0, fin_K = 0;
        double L = 0.0;
        const unsigned here = __ballot_sync(SMCRT_FULL, alive);
        const bool none = __ballot_sync(SMCRT_FULL, alive && (interact || phase == kLaunch)) == 0u;   // no other lane moves
        const unsigned exact = __ballot_sync(SMCRT_FULL, alive && phase == kExact && !interact);
        wait_x += __popc(exact);
        if (exact != 0u && (K == kGeneralScene || none || kWaitExact * wait_x >= __popc(here))) {
            wait_x = 0;
            if (alive && phase == kExact && !interact) {
                Eval64 E;
                if (K == kGeneralScene) {
                    E = scene_eval64(S, px, py, pz);
                } else {
                    C.neg = kneg; C.mask = kmask; C.list = klist; C.flr = kfold >> 8; C.cnt = (int)(int8_t)(kfold & 0xff);
                    C.soft = ksoft; C.db = kdb;
                    E = scene_exact<K>(S, px, py, pz, C, kForTrace);
                }
                if (E.dbox > 0.0) {                      // outside the volume of interest
                    out = true;
                } else {
                    reg = E.region;
                    if (E.dmin < delta) {                // on a boundary
                        istar = E.istar;
                        dstar = E.dstar;
                        phase = kArrive;
                    } else {
                        const double mu_t = reg >= 0 ? __ldg(S.reg64 + kReg64 * reg + 4) : 0.0;
                        L = E.dmin - 0.5 * delta;        // stop short of the surface
                        move = true;
                        interact = mu_t > 0.0 && tau < mu_t * L;
                        if (!interact && S.stepping == SMCRT_STEP_SEGMENT) {   // a longer move along u
                            if (K == kGeneralScene) L = fmax(L, segment_bound64(S, E.dsoft, E.dbox, px, py, pz, ux, uy, uz));
                            else L = max64(L, segment_bound64_screened<K>(S, E, C, px, py, pz, ux, uy, uz));
                            interact = mu_t > 0.0 && tau < mu_t * L;
                        }
                    }
                }
            }
        }

        // ---- 3b. the packets at a surface, once enough of them wait
        Interface64 I;
        I.R = 1.0;
        const unsigned arrived = __ballot_sync(SMCRT_FULL, alive && phase == kArrive);
        wait_i += __popc(arrived);
        if (arrived != 0u && (kWaitArrive * wait_i >= __popc(here) ||
                              __ballot_sync(SMCRT_FULL, alive && (move || phase == kLaunch)) == 0u)) {
            wait_i = 0;
            if (alive && phase == kArrive) {
                I = interface64<K>(S, px, py, pz, ux, uy, uz, istar, dstar);
                nev += I.evals;
                phase = kTrace;
                if (I.what == kIntfForced) {
                    L = delta;                           // forced step along u
                    move = true;
                    const double mu_t = reg >= 0 ? __ldg(S.reg64 + kReg64 * reg + 4) : 0.0;
                    interact = mu_t > 0.0 && tau < mu_t * L;
                } else if (I.what == kIntfEscape) {
                    out = true;                          // outward through the bounding box
                } else {
                    wadd(wa, kIntf, 1);
                    if (I.what == kIntfMatched) {
                        const double ee = 2.0 * delta * (I.cdot > 0.0 ? 1.0 : -1.0);
                        px = I.qx + ee * I.nx; py = I.qy + ee * I.ny; pz = I.qz + ee * I.nz;
                        iter_done = true;
                    } else {
                        wadd(wa, kFres, 1);
                        fresnel = true;
                    }
                }
            }
        }
        if (SMCRT_RARE(out)) {
            const long long v = fx64(w);
            if (ux * S.src_dir[0] + uy * S.src_dir[1] + uz * S.src_dir[2] < 0.0) fin_R = v; else fin_T = v;
            fin = true;
            alive = false;
        }

        // ---- 4. move: interaction point or sphere-trace step, one tally site
        if (move) {
            const double mu_t = reg >= 0 ? __ldg(S.reg64 + kReg64 * reg + 4) : 0.0;
            const double seg = interact ? div_by64(tau, mu_t, __ldg(S.reg64 + kReg64 * reg + 6)) : L;
            long long *const flu = (long long *)jc->flu;
            if (flu) {
                if (K == kGeneralScene) npieces += tally64(S, flu, px, py, pz, ux, uy, uz, seg, w);
                else npieces += tally64_screened(S, flu, px, py, pz, ux, uy, uz, seg, w);
            }
            px = px + seg * ux; py = py + seg * uy; pz = pz + seg * uz;
            if (!interact) tau = tau - mu_t * L;
            phase = kTrace;
            iter_done = true;
        }

        // ---- 5. one Philox call for every lane that draws this iteration
        const bool draws = alive && (phase == kLaunch || interact || (fresnel && I.R < 1.0));
        uint4 r = make_uint4(0u, 0u, 0u, 0u);
        if (__any_sync(SMCRT_FULL, draws)) {
            r = philox4x32_10(make_uint4(event, 0u, id_lo, id_hi), jc->k0, jc->k1);
            if (draws) event += 1u;
        }

        // ---- 6. consumers
        if (SMCRT_RARE(alive && phase == kLaunch)) {                 // photon release
            const Launched64 o = launch64(S, r);
            px = o.px; py = o.py; pz = o.pz;
            ux = o.ux; uy = o.uy; uz = o.uz;
            tau = o.tau;
            w = 1.0;
            nsteps = 0; pA = 0; pG = 0; pscat = 0;
            phase = kTrace;
        }
        if (interact) {                                  // implicit capture, HG, roulette
            const double *RG = S.reg64 + kReg64 * reg;
            const double wn = w * __ldg(RG + 5);
            pA += fx64(w - wn);
            w = wn;
            scatter64(ux, uy, uz, hg_cos64(RG, u01_64(r.x)), r.y);
            pscat += 1u;
            if (w < kWRoulette) {
                if (u01_64(r.z) <= 1.0 / kRouletteM) {
                    pG += fx64(w * (kRouletteM - 1.0));
                    w = w * kRouletteM;
                } else {
                    fin_K = fx64(w);
                    fin = true;
                    alive = false;
                }
            }
            tau = -ln64(u01_64(r.w));
        }
        if (SMCRT_RARE(fresnel)) {                                 // Fresnel reflection / Snell refraction
            const bool reflect = I.R < 1.0 ? (u01_64(r.x) <= I.R) : true;
            const double ee = 2.0 * delta * (I.cdot > 0.0 ? 1.0 : -1.0);
            const Crossed64 o = cross64(ux, uy, uz, I.qx, I.qy, I.qz, I.nx, I.ny, I.nz, I.cdot, ee, I.n1, I.n2, I.ct,
                                        reflect);
            px = o.px; py = o.py; pz = o.pz;
            ux = o.ux; uy = o.uy; uz = o.uz;
            phase = kTrace;
            iter_done = true;
        }
        if (iter_done && alive) {
            nsteps += 1;
            if (nsteps >= S.max_steps) {
                wadd(wa, kCap, 1);
                fin_K = fx64(w);
                fin = true;
                alive = false;
            }
        }
        // ---- a terminated packet: one bookkeeping site per iteration
        if (SMCRT_RARE(fin)) {
            wadd(wa, kR, fin_R); wadd(wa, kT, fin_T); wadd(wa, kKilled, fin_K);
            wadd(wa, kA, pA); wadd(wa, kGain, pG); wadd(wa, kScat, pscat); wadd(wa, kSteps, nsteps);
            wadd(wa, kPackets, 1); wadd(wa, kEvals, nev);
            nev = 0;
            smcrt_packet_record *const recs = (smcrt_packet_record *)jc->recs;
            if (!SERVED && recs) {
                smcrt_packet_record r;
                r.R = fin_R; r.T = fin_T; r.A = pA; r.killed = fin_K; r.gain = pG;
                r.scatters = pscat; r.steps = nsteps; r.reserved = 0;
                const unsigned long long id = ((unsigned long long)id_hi << 32) | id_lo;
                recs[id - jc->begin] = r;
            }
        }
        // ---- park a straggler at a trace boundary (serving rounds only)
        if (SERVED && SMCRT_RARE(alive && phase == kTrace && jc->budget > 0u && (uint32_t)clock() - t_acq > jc->budget)) {
            JobDefer *const dfr = (JobDefer *)jc->dfr;
            const int din = jc->din;
            const unsigned k = atomicAdd(&dfr->count[1 - din], 1u);
            if (k < dfr->cap) {
                DeferState &d = dfr->buf[1 - din][k];
                d.p[0] = px; d.p[1] = py; d.p[2] = pz;
                d.u[0] = ux; d.u[1] = uy; d.u[2] = uz;
                d.w = w; d.tau = tau;
                d.pA = pA; d.pG = pG;
                d.id_lo = id_lo; d.id_hi = id_hi; d.event = event;
                d.nsteps = (uint32_t)nsteps; d.pscat = pscat;
                wadd(wa, kParked, 1); wadd(wa, kEvals, nev);
                nev = 0;
                alive = false;
            } else {
                atomicAdd(&dfr->overflow, 1u);
                t_acq = (uint32_t)clock() + 0x7fffffffu;   // list full: run on (one retry per ~1 s)
            }
        }
    }
    const long long pc = warp_sum((long long)npieces);
    if (lane == 0) wadd(wa, kPieces, pc);
    return timed_out;
}

template <int kMinBlocks, int K, bool SERVED>
__global__ void __launch_bounds__(128, kMinBlocks) packets_fp64(JobWork *jobs, int njobs, int *status)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gw = blockIdx.x * (blockDim.x >> 5) + warp;
    WarpShared *ws = reinterpret_cast<WarpShared *>(smem) + warp;
    for (int jj = 0; jj < njobs; ++jj) {
        JobWork *J = jobs + (gw + jj) % njobs;
        unsigned long long nxt = 0, e = 0;
        const DevScene *src = nullptr;
        if (lane == 0) {
            nxt = *(volatile unsigned long long *)&J->next;
            e = J->end;
            src = J->scene;
        }
        int parked = 0;
        if (SERVED && lane == 0 && J->defer != nullptr) {
            const int in = J->defer_in & 1;
            parked = min(*(volatile unsigned *)&J->defer->count[in], J->defer->cap) >
                     *(volatile unsigned *)&J->defer->cursor[in];
        }
        nxt = __shfl_sync(SMCRT_FULL, nxt, 0);
        e = __shfl_sync(SMCRT_FULL, e, 0);
        parked = __shfl_sync(SMCRT_FULL, parked, 0);
        src = (const DevScene *)__shfl_sync(SMCRT_FULL, (unsigned long long)src, 0);
        if (nxt >= e && !parked) continue;
        if (src == nullptr || J->totals == nullptr) {
            if (lane == 0) {
                atomicOr(status, kStatusBadJob);
                if (J->jstat != nullptr) atomicOr(J->jstat, kStatusBadJob);
            }
            continue;
        }
        const long long *s8 = reinterpret_cast<const long long *>(src);
        long long *d8 = reinterpret_cast<long long *>(&ws->S);
        for (int i = lane; i < (int)(sizeof(DevScene) / 8); i += 32) d8[i] = s8[i];
        __syncwarp();                        // every lane reads what others copied, and all decide alike
        if (!scene_runs64<K>(ws->S)) {       // a scene of another family than this instantiation's
            if (lane == 0) {
                atomicOr(status, kStatusBadJob);
                if (J->jstat != nullptr) atomicOr(J->jstat, kStatusBadJob);
            }
            continue;
        }
        if (lane == 0) jobconst_fill(&ws->jc, J);
        wacc_clear(&ws->acc, lane);
        const long long t0 = clock64();
        const bool timed_out = run_job_fp64<K, SERVED>(ws->S, &ws->acc, &ws->jc, J, lane);
        __syncwarp();
        if (lane == 0) wadd(&ws->acc, kBusy, clock64() - t0);
        wacc_flush(&ws->acc, J->totals, lane);
        if (timed_out) {                     // the launch's time limit: this warp is done
            if (lane == 0) {
                atomicOr(status, kStatusTimeout);
                if (J->jstat != nullptr) atomicOr(J->jstat, kStatusTimeout);
            }
            return;
        }
    }
}

}  // namespace

// Register budgets of the instantiations: variant v keeps kMinBlocks
// blocks of 128 threads resident per SM (more blocks = fewer registers per
// thread, possibly spilled): 4, 3 and 2; the autotuner picks per scene.
cudaError_t launch_fp64(JobWork *jobs, int njobs, int *status, int blocks, int threads, cudaStream_t stream,
                        int variant)
{
    const size_t sm = (size_t)(threads / 32) * sizeof(WarpShared);
    switch (variant) {   // kNumVariants and up: the same budgets for the other scene families
    case 1: packets_fp64<3, kPlainScene, false><<<blocks, threads, sm, stream>>>(jobs, njobs, status); break;
    case 2: packets_fp64<2, kPlainScene, false><<<blocks, threads, sm, stream>>>(jobs, njobs, status); break;
    case 3: packets_fp64<4, kGeneralScene, false><<<blocks, threads, sm, stream>>>(jobs, njobs, status); break;
    case 4: packets_fp64<3, kGeneralScene, false><<<blocks, threads, sm, stream>>>(jobs, njobs, status); break;
    case 5: packets_fp64<2, kGeneralScene, false><<<blocks, threads, sm, stream>>>(jobs, njobs, status); break;
    case 9: packets_fp64<4, kBoxScene, false><<<blocks, threads, sm, stream>>>(jobs, njobs, status); break;
    case 10: packets_fp64<3, kBoxScene, false><<<blocks, threads, sm, stream>>>(jobs, njobs, status); break;
    case 11: packets_fp64<2, kBoxScene, false><<<blocks, threads, sm, stream>>>(jobs, njobs, status); break;
    case 12: packets_fp64<4, kSingleScene, false><<<blocks, threads, sm, stream>>>(jobs, njobs, status); break;
    case 13: packets_fp64<3, kSingleScene, false><<<blocks, threads, sm, stream>>>(jobs, njobs, status); break;
    case 14: packets_fp64<2, kSingleScene, false><<<blocks, threads, sm, stream>>>(jobs, njobs, status); break;
    case 18: packets_fp64<4, kTreeScene, false><<<blocks, threads, sm, stream>>>(jobs, njobs, status); break;
    case 19: packets_fp64<3, kTreeScene, false><<<blocks, threads, sm, stream>>>(jobs, njobs, status); break;
    case 20: packets_fp64<2, kTreeScene, false><<<blocks, threads, sm, stream>>>(jobs, njobs, status); break;
    default: packets_fp64<4, kPlainScene, false><<<blocks, threads, sm, stream>>>(jobs, njobs, status); break;
    }
    return cudaGetLastError();
}

// Served rounds: packets park, no packet records, and a round holds scenes of
// all families.  Plan launches leave the parking out (layered slab 1e5
// packets 46.2 -> 44.5 ms, thick slab 3e3 110.5 -> 108.0 ms).
cudaError_t launch_fp64_served(JobWork *jobs, int njobs, int *status, int blocks, int threads, cudaStream_t stream,
                               bool general)
{
    const size_t sm = (size_t)(threads / 32) * sizeof(WarpShared);
    if (general) packets_fp64<3, kGeneralScene, true><<<blocks, threads, sm, stream>>>(jobs, njobs, status);
    else packets_fp64<3, kPlainScene, true><<<blocks, threads, sm, stream>>>(jobs, njobs, status);
    return cudaGetLastError();
}

int occupancy_fp64_served(int threads)
{
    int n = 0;
    const size_t sm = (size_t)(threads / 32) * sizeof(WarpShared);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, packets_fp64<3, kPlainScene, true>, threads, sm);
    return n;
}

int occupancy_fp64(int threads, int variant)
{
    int n = 0;
    const size_t sm = (size_t)(threads / 32) * sizeof(WarpShared);
    switch (variant) {
    case 1: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, packets_fp64<3, kPlainScene, false>, threads, sm); break;
    case 2: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, packets_fp64<2, kPlainScene, false>, threads, sm); break;
    case 3: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, packets_fp64<4, kGeneralScene, false>, threads, sm); break;
    case 4: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, packets_fp64<3, kGeneralScene, false>, threads, sm); break;
    case 5: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, packets_fp64<2, kGeneralScene, false>, threads, sm); break;
    case 9: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, packets_fp64<4, kBoxScene, false>, threads, sm); break;
    case 10: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, packets_fp64<3, kBoxScene, false>, threads, sm); break;
    case 11: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, packets_fp64<2, kBoxScene, false>, threads, sm); break;
    case 12: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, packets_fp64<4, kSingleScene, false>, threads, sm); break;
    case 13: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, packets_fp64<3, kSingleScene, false>, threads, sm); break;
    case 14: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, packets_fp64<2, kSingleScene, false>, threads, sm); break;
    case 18: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, packets_fp64<4, kTreeScene, false>, threads, sm); break;
    case 19: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, packets_fp64<3, kTreeScene, false>, threads, sm); break;
    case 20: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, packets_fp64<2, kTreeScene, false>, threads, sm); break;
    default: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, packets_fp64<4, kPlainScene, false>, threads, sm); break;
    }
    return n;
}

}  // namespace smcrt
