// duo.cuh - the two-warp layouts of the SRB rollout (arxiv 2603.20525, Sec.
// IV-A..IV-D), shared by the planning kernels and the adjoint's forward pass.
#pragma once

#include <cuda_runtime.h>
#include <math_constants.h>
#include <stdint.h>

#include "adjoint.cuh"
#include "atp.h"
#include "plan_kernel.cuh"
#include "plan_tail.cuh"
#include "srb_model.cuh"

namespace atp {

// ACC selects the running cost's accumulator: kAccF32, kAccF64, or
// kAccRuntime (p.acc64 decides; the batch kernel, which would otherwise inline
// twice as many variants).  A compile-time choice keeps the step loop free of
// the uniform branch.
constexpr int kAccF32 = 0, kAccF64 = 1, kAccRuntime = 2;

// ---- two warps per group of candidates ------------------------------------
//
// Forward Euler moves position and attitude with the velocities of the step's
// start, so the lookups of step t + 1 do not wait for the forces of step t.
// In each pair of warps one ("geometry") advances position, attitude and
// steering and looks the terrain up, and the other ("forces") turns the
// geometry of step t into the velocities of step t + 1, and accumulates the
// cost and the margins, while the first is at the geometry of step t + 1.
// They swap through shared memory (two buffers) with one CTA barrier per Euler
// step:
//
//   slot t    geometry warp: v(t) -> state(t+1) -> geometry(t+1)
//             forces warp:   geometry(t), v(t) -> v(t+1)
//
// Every quantity is formed by the same expressions as in one thread, so the
// bits are the same.

// What a rollout keeps for the adjoint (NoTrace: nothing, a plan).  It then
// runs control steps [k0, k1) from the checkpoint `from` (or from the start
// state), writes the Euler-step start states of [trace_k0, k1) that are
// executed, and every `seg` control steps a checkpoint.  A record is four
// float4: (x, xl, y, yl), (z, zl, psi, theta), (phi, delta, vx, vy),
// (vz, wx, wy, wz).  The force sums take the adjoint's own order.
struct NoTrace {
    static constexpr bool on = false;
};
struct Trace {
    static constexpr bool on = true;
    int k0, k1, trace_k0, seg;
    int objective;            // kGradCost or kGradMargin
    float4 *rec;              // [K][(k1 - trace_k0) n_sub][4]
    const float *from;        // [20][K] or nullptr: the state at k0
    float *ckpt;              // [ceil(H / seg)][20][K] or nullptr
    int *n_done;              // [K] Euler steps executed (written by a pass from step 0)
    int *emin;                // [K] index of the state holding the margin
    float4 *fin;              // [K] final x and y from the goal, theta, phi
};

// index in tr.rec of candidate j's record of step k0 n_sub (before the trace
// while k0 < trace_k0)
__device__ __forceinline__ long long first_record(const Trace &tr, int n_sub, int j)
{
    return ((long long)j * (tr.k1 - tr.trace_k0) + (tr.k0 - tr.trace_k0)) * n_sub * 4;
}

template <int LANES>
struct Duo {
    static constexpr int kW = 4 / LANES;            // wheels per lane
    static constexpr int kC = 32 / LANES;           // candidates per pair of warps
    float4 ground[2][kW][32];                       // WheelGround per wheel
    float4 att[2][kC];                              // sin and cos of theta, then of phi
    float2 yaw[2][kC];                              // sin and cos of psi
    float4 body[2][kC];                             // delta, cos(delta), phi; done (0 or 1)
    float4 va[2][kC];                               // vx, vy, vz, wx
    float2 vb[2][kC];                               // wy, wz
    float d2[kC];                                   // final squared distance to the goal
    int flags[kC];                                  // done, off the map, final state not finite
    int flip;                                       // which warp takes which role
};

constexpr unsigned kFull = 0xffffffffu;

// c ? a : b as a select: the compiler turns chains of conditionals on the
// lane into divergent branches, which cost far more than the selects
__device__ __forceinline__ float sel(bool c, float a, float b)
{
    float r;
    asm("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %3, 0;\n\tselp.f32 %0, %1, %2, p;\n\t}" : "=f"(r) : "f"(a), "f"(b), "r"((int)c));
    return r;
}
__device__ __forceinline__ void pair_barrier() { asm volatile("bar.sync 0;" ::: "memory"); }

// this lane's first wheel or axle
struct LaneWheel {
    bool front;
    float rx, ry, k, b, Fs;
};
template <int LANES>
__device__ __forceinline__ LaneWheel lane_wheel(const Veh &V, int q)
{
    LaneWheel w;
    w.front = LANES == 1 || (LANES == 2 ? q == 0 : q < 2);
    w.rx = w.front ? V.Lf : -V.Lr;
    w.ry = LANES < 4 ? V.he : (q & 1) ? -V.he : V.he;
    w.k = w.front ? V.kf : V.kr;
    w.b = w.front ? V.bf : V.br;
    w.Fs = w.front ? V.Fsf : V.Fsr;
    return w;
}

// Sum of v over the two lanes of a candidate's pair (a0 + a1 in both).
__device__ __forceinline__ float pair_sum(float v) { return v + __shfl_xor_sync(kFull, v, 1); }
// sum over the four lanes of a candidate (the same bits in every lane)
__device__ __forceinline__ float quad_sum(float v)
{
    v += __shfl_xor_sync(kFull, v, 1);
    return v + __shfl_xor_sync(kFull, v, 2);
}

// Two neighbouring float4 of a record, by two lanes where there are two.
template <int LANES>
__device__ __forceinline__ void put_record(const Trace &tr, long long at, int q, float4 a, float4 b)
{
    if constexpr (LANES == 1) {
        tr.rec[at] = a;
        tr.rec[at + 1] = b;
    } else {
        const bool o = q != 0;
        const float4 v = make_float4(sel(o, b.x, a.x), sel(o, b.y, a.y), sel(o, b.z, a.z), sel(o, b.w, a.w));
        if (q < 2) tr.rec[at + q] = v;
    }
}

struct Fast { static constexpr bool value = false; };
struct Slow { static constexpr bool value = true; };

template <int LANES, bool PER_X0, int TEX, class Tr>
__device__ __forceinline__ void duo_geometry(const PlanParams &p, const Tr &tr, Duo<LANES> &sh, int j, int q, int c,
                                             bool live)
{
    const Veh &V = p.V;
    const Cost &Cc = p.C;
    const Terrain &T = p.T;
    const int lane = threadIdx.x & 31;
    const LaneWheel lw = lane_wheel<LANES>(V, q);
    float x = 0.f, xl = 0.f, y = 0.f, yl = 0.f, z = 0.f, zl = 0.f, psi = 0.f, psil = 0.f, th = 0.f, ph = 0.f, d = 0.f;
    if (live) {
        const size_t N = (size_t)p.N;
        const auto x0 = [&](int r) { return PER_X0 ? __ldg(p.x0_soa + r * N + j) : p.x0[r]; };
        two_sum(x0(0), -T.x0_hi, x, xl);
        xl -= T.x0_lo;
        two_sum(x0(1), -T.y0_hi, y, yl);
        yl -= T.y0_lo;
        z = x0(2); psi = x0(3); th = x0(4); ph = x0(5); d = x0(12);
    }
    bool done = !live, off = false, offs = false;
    int k_begin = 0, k_end = p.H, n_exec = 0;
    [[maybe_unused]] long long rec = 0;
    if constexpr (Tr::on) {
        k_begin = tr.k0;
        k_end = tr.k1;
        rec = first_record(tr, p.n_sub, j);
        if (live && tr.from) {
            const size_t N = (size_t)p.N;
            const auto ck = [&](int r) { return tr.from[r * N + j]; };
            x = ck(0); xl = ck(1); y = ck(2); yl = ck(3); z = ck(4); zl = ck(5); psi = ck(6); psil = ck(7);
            th = ck(8); ph = ck(9); d = ck(10);
        }
    }
    const float h = p.h;
    float R[9], sth = 0.f, cth = 1.f, sph = 0.f, cph = 1.f;
    const bool q1 = (q & 1) != 0, q2 = (q & 2) != 0;
    bool huge = false;               // an angle beyond the fast reduction

    // the goal test and the wheels' geometry of the current state, into
    // buffer `par`
    const auto geometry = [&](int par, auto form) {
        float sps, cps, cdl;
        if constexpr (LANES == 4) {
            float s1, c1;
            const float an = sel(q2, sel(q1, d, ph), sel(q1, th, psi));
            sincos_g<decltype(form)::value>(an, s1, c1);
            huge = fabsf(an) >= kSincosMax;
            sps = __shfl_sync(kFull, s1, 0, 4);
            cps = __shfl_sync(kFull, c1, 0, 4);
            sth = __shfl_sync(kFull, s1, 1, 4);
            cth = __shfl_sync(kFull, c1, 1, 4);
            sph = __shfl_sync(kFull, s1, 2, 4);
            cph = __shfl_sync(kFull, c1, 2, 4);
            cdl = __shfl_sync(kFull, c1, 3, 4);
        } else if constexpr (LANES == 1) {
            float sdl;
            sincos_g<decltype(form)::value>(psi, sps, cps);
            sincos_g<decltype(form)::value>(th, sth, cth);
            sincos_g<decltype(form)::value>(ph, sph, cph);
            sincos_g<decltype(form)::value>(d, sdl, cdl);
            huge = fmaxf(fmaxf(fabsf(psi), fabsf(th)), fmaxf(fabsf(ph), fabsf(d))) >= kSincosMax;
        } else {
            // lane 0: psi and phi; lane 1: theta and delta
            float s1, c1, s2, c2;
            const float a1 = sel(q1, th, psi), a2 = sel(q1, d, ph);
            sincos_g<decltype(form)::value>(a1, s1, c1);
            sincos_g<decltype(form)::value>(a2, s2, c2);
            huge = fmaxf(fabsf(a1), fabsf(a2)) >= kSincosMax;
            const float os1 = __shfl_xor_sync(kFull, s1, 1), oc1 = __shfl_xor_sync(kFull, c1, 1);
            const float os2 = __shfl_xor_sync(kFull, s2, 1), oc2 = __shfl_xor_sync(kFull, c2, 1);
            sps = sel(q1, os1, s1);
            cps = sel(q1, oc1, c1);
            sth = sel(q1, s1, os1);
            cth = sel(q1, c1, oc1);
            sph = sel(q1, os2, s2);
            cph = sel(q1, oc2, c2);
            cdl = sel(q1, c2, oc2);
        }
        rotation(sps, cps, sth, cth, sph, cph, R);
        // goal test before the step (Sec. IV-C, reading Q4)
        const float gdx = (x - Cc.gx_hi) + (xl - Cc.gx_lo);
        const float gdy = (y - Cc.gy_hi) + (yl - Cc.gy_lo);
        done = done || fmaf(gdx, gdx, gdy * gdy) <= Cc.goal_r2;
        if (q == 0) {
            sh.att[par][c] = make_float4(sth, cth, sph, cph);
            sh.yaw[par][c] = make_float2(sps, cps);
            sh.body[par][c] = make_float4(d, cdl, ph, done ? 1.f : 0.f);
        }
        const Cell cx = cell_of<!Tr::on>(x, xl, T.inv_cell, T.nx), cy = cell_of<!Tr::on>(y, yl, T.inv_cell, T.ny);
        const unsigned base = texel_base(cx, cy, T.nx);
        offs = off_com(cx, cy);
    #pragma unroll
        for (int w = 0; w < Duo<LANES>::kW; ++w) {
            const WheelGround g = wheel_ground<TEX>(V, T, R, cx, cy, base, z, zl, w < 2 ? lw.rx : -V.Lr,
                                                    LANES == 4 ? lw.ry : (w & 1) ? -V.he : V.he, offs);
            sh.ground[par][w][lane] = make_float4(g.fx, g.fy, g.Q, g.cost);
        }
    };

    geometry(0, Fast{});
    if (__any_sync(kFull, huge)) geometry(0, Slow{});
    pair_barrier();
    int par = 0;
    float un = live ? __ldg(&p.ctrl[(size_t)k_begin * p.N + j].x) : 0.f;
    for (int k = k_begin; k < k_end; ++k) {
        // zero-order hold; admissible steering rate |delta_dot| <= max
        const float dd = clamp_keep_nan(un, -V.ddmax, V.ddmax);
        if constexpr (Tr::on) {
            if (tr.ckpt && k % tr.seg == 0 && live && q == 0) {
                const size_t N = (size_t)p.N;
                float *o = tr.ckpt + (size_t)(k / tr.seg) * 20 * N + j;
                const float v[11] = {x, xl, y, yl, z, zl, psi, psil, th, ph, d};
#pragma unroll
                for (int r = 0; r < 11; ++r) o[r * N] = v[r];
            }
        }
        if (live && k + 1 < k_end) un = __ldg(&p.ctrl[(size_t)(k + 1) * p.N + j].x);
        const bool idle = __all_sync(kFull, done);     // every candidate frozen at the goal
        for (int sub = 0; sub < p.n_sub; ++sub) {
            if (!idle) {
                const float4 va = sh.va[par][c];
                const float2 vb = sh.vb[par][c];
                const float vx = va.x, vy = va.y, vz = va.z, wx = va.w, wy = vb.x, wz = vb.y;
                const bool go = !done;
                off = off || (go && offs);
                if constexpr (Tr::on) {
                    if (go && k >= tr.trace_k0)
                        put_record<LANES>(tr, rec, q, make_float4(x, xl, y, yl), make_float4(z, zl, psi, th));
                    n_exec += go ? 1 : 0;
                }
                // position, attitude and steering of A(xi) + B zeta (Sec. IV-A), forward Euler
                const float ic = rcp(cth);
                const float wsc = fmaf(sph, wy, cph * wz);
                const float dx = fmaf(R[2], vz, fmaf(R[1], vy, R[0] * vx));
                const float dy = fmaf(R[5], vz, fmaf(R[4], vy, R[3] * vx));
                const float dz = fmaf(R[8], vz, fmaf(R[7], vy, R[6] * vx));
                const float dpsi = wsc * ic;
                const float dth = fmaf(cph, wy, -sph * wz);
                const float dph = fmaf(wsc, sth * ic, wx);
                float nx = x, nxl = xl, ny = y, nyl = yl, nz = z, nzl = zl, np_ = psi, npl = psil;
                acc2(nx, nxl, h * dx);
                acc2(ny, nyl, h * dy);
                acc2(nz, nzl, h * dz);
                acc2(np_, npl, h * dpsi);
                const float nth = fmaf(h, dth, th), nph = fmaf(h, dph, ph);
                const float nd = clamp_keep_nan(fmaf(h, dd, d), -V.dmax, V.dmax);
                // frozen at the goal: the step is computed and discarded, which
                // keeps the warp converged for the shuffles
                x = sel(go, nx, x); xl = sel(go, nxl, xl); y = sel(go, ny, y); yl = sel(go, nyl, yl);
                z = sel(go, nz, z); zl = sel(go, nzl, zl); psi = sel(go, np_, psi); psil = sel(go, npl, psil);
                th = sel(go, nth, th); ph = sel(go, nph, ph); d = sel(go, nd, d);
                geometry(par ^ 1, Fast{});
                if (__any_sync(kFull, huge)) geometry(par ^ 1, Slow{});
            }
            pair_barrier();
            par ^= 1;
            if constexpr (Tr::on) rec += 4;
        }
    }
    if constexpr (Tr::on) {
        // the forces warp ends the objective with these
        if (q == 0) {
            const float gdx = (x - Cc.gx_hi) + (xl - Cc.gx_lo);
            const float gdy = (y - Cc.gy_hi) + (yl - Cc.gy_lo);
            sh.d2[c] = fmaf(gdx, gdx, gdy * gdy);
            sh.flags[c] = n_exec;
            if (live && tr.k0 == 0 && k_end == p.H) {
                tr.n_done[j] = n_exec;
                tr.fin[j] = make_float4(gdx, gdy, th, ph);
            }
        }
        pair_barrier();
        return;
    }
    // the off-map flag is per wheel: OR it over the candidate's lanes
    const unsigned offm = __ballot_sync(kFull, off) >> (lane & ~(LANES - 1));
    off = (offm & ((1u << LANES) - 1u)) != 0u;
    // fold the low parts back and leave the terrain frame
    const float xs[7] = {(x + T.x0_hi) + (xl + T.x0_lo), (y + T.y0_hi) + (yl + T.y0_lo), z + zl, psi + psil, th, ph,
                         d};
    if (q == 0) {
        const float gdx = (x - Cc.gx_hi) + (xl - Cc.gx_lo);
        const float gdy = (y - Cc.gy_hi) + (yl - Cc.gy_lo);
        bool finite = true;
#pragma unroll
        for (int r = 0; r < 7; ++r) finite = finite && isfinite(xs[r]);
        sh.d2[c] = fmaf(gdx, gdx, gdy * gdy);
        sh.flags[c] = (done ? ATP_FLAG_DONE : 0) | (off ? ATP_FLAG_OFFMAP : 0) | (finite ? 0 : ATP_FLAG_NONFINITE);
        if (live && p.xf) {
            const size_t N = (size_t)p.N;
#pragma unroll
            for (int r = 0; r < 6; ++r) p.xf[r * N + j] = xs[r];
            p.xf[12 * N + j] = xs[6];
        }
    }
    pair_barrier();
}

template <int LANES, bool PER_X0, int ACC, class Tr>
__device__ __forceinline__ void duo_forces(const PlanParams &p, const Tr &tr, Duo<LANES> &sh, int j, int q, int c, bool live,
                                           float &J, float &margin, bool &feasible)
{
    const Veh &V = p.V;
    const Cost &Cc = p.C;
    const int lane = threadIdx.x & 31;
    const LaneWheel lw = lane_wheel<LANES>(V, q);
    const bool front = lw.front, left = (q & 1) == 0;
    float vx = 0.f, vxl = 0.f, vy = 0.f, vyl = 0.f, vz = 0.f, vzl = 0.f, wx = 0.f, wy = 0.f, wz = 0.f;
    if (live) {
        const size_t N = (size_t)p.N;
        const auto x0 = [&](int r) { return PER_X0 ? __ldg(p.x0_soa + r * N + j) : p.x0[r]; };
        vx = x0(6); vy = x0(7); vz = x0(8); wx = x0(9); wy = x0(10); wz = x0(11);
    }
    int k_begin = 0, k_end = p.H, emin = 0;
    [[maybe_unused]] long long rec = 0;
    if constexpr (Tr::on) {
        k_begin = tr.k0;
        k_end = tr.k1;
        rec = first_record(tr, p.n_sub, j);
        if (live && tr.from) {
            const size_t N = (size_t)p.N;
            const auto ck = [&](int r) { return tr.from[r * N + j]; };
            vx = ck(11); vxl = ck(12); vy = ck(13); vyl = ck(14); vz = ck(15); vzl = ck(16);
            wx = ck(17); wy = ck(18); wz = ck(19);
        }
    }
    const float h = p.h;
    const bool acc64 = ACC == kAccRuntime ? p.acc64 != 0 : ACC == kAccF64;
    const bool cm = p.T.has_cm != 0;
    double J64 = 0.0;
    float U = 0.f, msm = CUDART_INF_F, last_sm = CUDART_INF_F;
    int mstep = 0;
    if (q == 0) {
        sh.va[0][c] = make_float4(vx, vy, vz, wx);
        sh.vb[0][c] = make_float2(wy, wz);
    }
    pair_barrier();
    int par = 0;
    bool idle = false;
    float2 un = live ? __ldg(p.ctrl + (size_t)k_begin * p.N + j) : make_float2(0.f, 0.f);
    for (int k = k_begin; k < k_end; ++k) {
        const float dd = clamp_keep_nan(un.x, -V.ddmax, V.ddmax), ax = un.y;
        if (live && k + 1 < k_end) un = __ldg(p.ctrl + (size_t)(k + 1) * p.N + j);
        if constexpr (Tr::on) {
            if (tr.ckpt && k % tr.seg == 0 && live && q == 0) {
                const size_t N = (size_t)p.N;
                float *o = tr.ckpt + ((size_t)(k / tr.seg) * 20 + 11) * N + j;
                const float v[9] = {vx, vxl, vy, vyl, vz, vzl, wx, wy, wz};
#pragma unroll
                for (int r = 0; r < 9; ++r) o[r * N] = v[r];
            }
        }
        if (!idle) {
            // for good: the geometry warp leaves the buffers as they are
            const float4 att = sh.att[par][c], body = sh.body[par][c];
            U = esm(V, body.z, att.z, att.w, att.y);
            idle = __all_sync(kFull, body.w != 0.f);
        }
        float sm = CUDART_INF_F;
        for (int sub = 0; sub < p.n_sub; ++sub) {
            if (!idle) {
                const float4 att = sh.att[par][c], body = sh.body[par][c];
                const float sth = att.x, cth = att.y, sph = att.z, cph = att.w, cd = body.y;
                const float di = front ? body.x : 0.f;
                const bool go = body.w == 0.f;
                if constexpr (Tr::on) {
                    if (go && k >= tr.trace_k0)
                        put_record<LANES>(tr, rec + 2, q, make_float4(body.z, body.x, vx, vy),
                                          make_float4(vz, wx, wy, wz));
                }
                // gravity in B: R^T (0, 0, -g)
                const float gBx = -V.g * -sth, gBy = -V.g * (cth * sph), gBz = -V.g * (cph * cth);
                // summed forces and moments (Sec. IV-A); the rear
                // longitudinal constraint force enters My only
                float FyB, FzB, Mx, My, Mz, csum = 0.f;
                // the rotation again, which the forces warp has time for
                const float2 yaw = sh.yaw[par][c];
                float R[9];
                rotation(yaw.x, yaw.y, sth, cth, sph, cph, R);
                const auto geo = [&](int w) {
                    const float4 t = sh.ground[par][w][lane];
                    return wheel_geo(R, WheelGround{t.x, t.y, t.z, t.w});
                };
                const WheelGeo g0 = geo(0);
                if constexpr (LANES == 1) {
                    const auto wh = [&](int i, float rx, float ry, float k, float b, float Fs, float dw) {
                        const WheelGeo g = i == 0 ? g0 : geo(i);
                        return wheel_dyn<false, Tr::on>(V, g, vx, vy, vz, wx, wy, wz, rx, ry, k, b, Fs, dw);
                    };
                    const WheelOut fl = wh(0, V.Lf, V.he, V.kf, V.bf, V.Fsf, di), fr = wh(1, V.Lf, -V.he, V.kf, V.bf, V.Fsf, di);
                    const WheelOut rl = wh(2, -V.Lr, V.he, V.kr, V.br, V.Fsr, 0.f), rr = wh(3, -V.Lr, -V.he, V.kr, V.br, V.Fsr, 0.f);
                    FzB = (fl.Fz + fr.Fz) + (rl.Fz + rr.Fz);
                    if constexpr (Tr::on) {
                        const float y0 = fl.Fy * cd, y1 = fr.Fy * cd;
                        FyB = (y0 + y1) + (rl.Fy + rr.Fy);
                        Mx = fmaf(V.hR, FyB, (V.he * fl.Fz + -V.he * fr.Fz) + (V.he * rl.Fz + -V.he * rr.Fz));
                        My = (-V.Lf * fl.Fz + -V.Lf * fr.Fz) + (V.Lr * rl.Fz + V.Lr * rr.Fz);
                        Mz = (V.Lf * y0 + V.Lf * y1) + (-V.Lr * rl.Fy + -V.Lr * rr.Fy);
                    } else {
                        const float Fyf = (fl.Fy + fr.Fy) * cd;
                        const float Fyr = rl.Fy + rr.Fy;
                        FyB = Fyf + Fyr;
                        Mx = fmaf(V.hR, FyB, V.he * ((fl.Fz - fr.Fz) + (rl.Fz - rr.Fz)));
                        My = -V.Lf * (fl.Fz + fr.Fz) + V.Lr * (rl.Fz + rr.Fz);
                        Mz = V.Lf * Fyf + -V.Lr * Fyr;
                    }
                    csum = (fl.cost + fr.cost) + (rl.cost + rr.cost);
                } else if constexpr (LANES == 2) {
                    const WheelGeo g1 = geo(1);
                    const WheelOut l = wheel_dyn<true, Tr::on>(V, g0, vx, vy, vz, wx, wy, wz, lw.rx, V.he, lw.k, lw.b, lw.Fs, di);
                    const WheelOut r = wheel_dyn<true, Tr::on>(V, g1, vx, vy, vz, wx, wy, wz, lw.rx, -V.he, lw.k, lw.b, lw.Fs, di);
                    FzB = pair_sum(l.Fz + r.Fz);
                    if constexpr (Tr::on) {
                        const float y0 = sel(front, l.Fy * cd, l.Fy), y1 = sel(front, r.Fy * cd, r.Fy);
                        FyB = pair_sum(y0 + y1);
                        Mx = fmaf(V.hR, FyB, pair_sum(V.he * l.Fz + -V.he * r.Fz));
                        My = pair_sum(-lw.rx * l.Fz + -lw.rx * r.Fz);
                        Mz = pair_sum(lw.rx * y0 + lw.rx * y1);
                    } else {
                        const float fy = sel(front, (l.Fy + r.Fy) * cd, l.Fy + r.Fy);
                        FyB = pair_sum(fy);
                        Mx = fmaf(V.hR, FyB, V.he * pair_sum(l.Fz - r.Fz));
                        My = pair_sum(-lw.rx * (l.Fz + r.Fz));
                        Mz = pair_sum(lw.rx * fy);
                    }
                    if (cm) csum = pair_sum(l.cost + r.cost);
                } else {
                    // the axle's sums by one xor-shuffle, the other axle's by a
                    // second, each formed in the order one lane forms it
                    const WheelOut w = wheel_dyn<false, Tr::on>(V, g0, vx, vy, vz, wx, wy, wz, lw.rx, lw.ry, lw.k, lw.b, lw.Fs, di);
                    if constexpr (Tr::on) {
                        const float fy = sel(front, w.Fy * cd, w.Fy);
                        FyB = quad_sum(fy);
                        FzB = quad_sum(w.Fz);
                        Mx = fmaf(V.hR, FyB, quad_sum(lw.ry * w.Fz));
                        My = quad_sum(-lw.rx * w.Fz);
                        Mz = quad_sum(lw.rx * fy);
                    } else {
                        const float oFy = __shfl_xor_sync(kFull, w.Fy, 1);
                        const float oFz = __shfl_xor_sync(kFull, w.Fz, 1);
                        const float aFy = w.Fy + oFy;
                        const float afy = sel(front, aFy * cd, aFy);               // Fyf or Fyr
                        const float aFz = w.Fz + oFz;
                        const float aDz = sel(left, w.Fz - oFz, oFz - w.Fz);        // left - right
                        const float bfy = __shfl_xor_sync(kFull, afy, 2);
                        const float bFz = __shfl_xor_sync(kFull, aFz, 2);
                        const float bDz = __shfl_xor_sync(kFull, aDz, 2);
                        const float Fyf = sel(front, afy, bfy), Fyr = sel(front, bfy, afy);
                        const float Fzf = sel(front, aFz, bFz), Fzr = sel(front, bFz, aFz);
                        FyB = Fyf + Fyr;
                        FzB = Fzf + Fzr;
                        Mx = fmaf(V.hR, FyB, V.he * (aDz + bDz));
                        My = -V.Lf * Fzf + V.Lr * Fzr;
                        Mz = V.Lf * Fyf + -V.Lr * Fyr;
                    }
                    if (cm) {
                        const float ac = w.cost + __shfl_xor_sync(kFull, w.cost, 1);
                        csum = ac + __shfl_xor_sync(kFull, ac, 2);
                    }
                }
                const float Fx = V.halfM * fmaf(-wz, vy, fmaf(wy, vz, ax - gBx));
                My = fmaf(-V.hR, 2.f * Fx, My);
                // the velocity rows of A(xi) + B zeta (Sec. IV-A), forward Euler
                const float dvy = fmaf(-wz, vx, fmaf(wx, vz, fmaf(FyB, V.invM, gBy)));
                const float dvz = fmaf(wy, vx, fmaf(-wx, vy, fmaf(FzB, V.invM, gBz)));
                const float dwx = fmaf(V.dJyz * wy, wz, Mx) * V.invJxx;
                const float dwy = fmaf(-V.dJxz * wx, wz, My) * V.invJyy;
                const float dwz = fmaf(V.dJxy * wx, wy, Mz) * V.invJzz;
                float nvx = vx, nvxl = vxl, nvy = vy, nvyl = vyl, nvz = vz, nvzl = vzl;
                acc2(nvx, nvxl, h * ax);
                acc2(nvy, nvyl, h * dvy);
                acc2(nvz, nvzl, h * dvz);
                const float nwx = fmaf(h, dwx, wx), nwy = fmaf(h, dwy, wy), nwz = fmaf(h, dwz, wz);
                vx = sel(go, nvx, vx); vxl = sel(go, nvxl, vxl); vy = sel(go, nvy, vy); vyl = sel(go, nvyl, vyl);
                vz = sel(go, nvz, vz); vzl = sel(go, nvzl, vzl);
                wx = sel(go, nwx, wx); wy = sel(go, nwy, wy); wz = sel(go, nwz, wz);
                if (q == 0) {
                    sh.va[par ^ 1][c] = make_float4(vx, vy, vz, wx);
                    sh.vb[par ^ 1][c] = make_float2(wy, wz);
                }
                // running cost L = L_0 + L_soft (Sec. IV-C), left Riemann sum
                U = esm(V, body.z, sph, cph, cth);
                if constexpr (Tr::on) {
                    if (U < margin) {            // the first state on ties
                        margin = U;
                        emin = k * p.n_sub + sub;
                    }
                } else {
                    margin = fminf(margin, U);
                }
                const float soft = fmaxf(fmaf(-U, Cc.inv_eps, 1.f), 0.f);
                const float L = fmaf(Cc.sigma * soft, soft, fmaf(Cc.wc * dd, dd, Cc.wt)) + csum;
                if (acc64) J64 += go ? (double)(h * L) : 0.0;
                else J = sel(go, fmaf(h, L, J), J);
            }
            sm = fminf(sm, U);
            pair_barrier();
            par ^= 1;
            if constexpr (Tr::on) rec += 4;
        }
        if (live && p.step_margin && q == 0 && k + 1 < p.H) p.step_margin[(size_t)k * p.N + j] = sm;
        if (k + 1 < p.H) {
            if (sm < msm) {
                msm = sm;
                mstep = k;
            }
        } else {
            last_sm = sm;
        }
    }
    pair_barrier();                       // the geometry warp's final state is stored
    if (!live) return;
    if constexpr (Tr::on) {
        if (tr.k0 != 0 || k_end != p.H) return;      // a segment again, for its trace
        if (!idle) {
            const float4 att = sh.att[par][c], body = sh.body[par][c];
            U = esm(V, body.z, att.z, att.w, att.y);
        }
        if (U < margin) {
            margin = U;
            emin = sh.flags[c];
        }
        if (q == 0) {
            tr.emin[j] = emin;
            p.cost[j] = tr.objective == kGradMargin ? margin : fmaf(Cc.wg, sqrtf(sh.d2[c]), J);
        }
        return;
    }
    // final state: margin and terminal cost Phi (Sec. IV-C)
    if (!idle) {
        const float4 att = sh.att[par][c], body = sh.body[par][c];
        U = esm(V, body.z, att.z, att.w, att.y);
    }
    margin = fminf(margin, U);
    last_sm = fminf(last_sm, U);
    if (last_sm < msm) mstep = p.H - 1;
    if (p.step_margin && q == 0) p.step_margin[(size_t)(p.H - 1) * p.N + j] = last_sm;
    const float d2 = sh.d2[c];
    if (acc64) J = (float)(J64 + (double)(Cc.wg * sqrtf(d2)));
    else J = fmaf(Cc.wg, sqrtf(d2), J);
    const float xs[6] = {vx + vxl, vy + vyl, vz + vzl, wx, wy, wz};
    const int gfl = sh.flags[c];
    bool finite = isfinite(J) && !(gfl & ATP_FLAG_NONFINITE);
#pragma unroll
    for (int r = 0; r < 6; ++r) finite = finite && isfinite(xs[r]);
    if (!finite) J = CUDART_INF_F;
    feasible = finite && margin > 0.f;
    if (q == 0) {
        const uint8_t fl = (feasible ? ATP_FLAG_FEASIBLE : 0) | (gfl & (ATP_FLAG_DONE | ATP_FLAG_OFFMAP)) |
                           (finite ? 0 : ATP_FLAG_NONFINITE);
        if (p.cost) p.cost[j] = J;
        if (p.margin) p.margin[j] = margin;
        if (p.flags) p.flags[j] = fl;
        if (p.min_step) p.min_step[j] = mstep;
        if (p.xf) {
            const size_t N = (size_t)p.N;
#pragma unroll
            for (int r = 0; r < 6; ++r) p.xf[(6 + r) * N + j] = xs[r];
        }
    }
}

// Whether this warp is its pair's geometry warp.  Warps w and w + 4 share an
// SM sub-partition, and the geometry warp issues about 1.3 times the forces
// warp's instructions: the roles alternate by the CTA's warp slots, so that
// the sub-partitions get both kinds (the scaled plan 407 -> 336 us with two
// lanes).  The shuffle makes the answer uniform over the warp, so that the
// branch on it is a plain jump (4 % of a small plan).
__device__ __forceinline__ bool geometry_role(int &flip)
{
    if (threadIdx.x == 0) {
        unsigned wid;
        asm volatile("mov.u32 %0, %%warpid;" : "=r"(wid));
        flip = (wid >> 2) & 1;
    }
    __syncthreads();
    return __shfl_sync(kFull, (int)(threadIdx.x >> 5) ^ flip, 0) == 0;
}

// One CTA of a two-warp plan; `cta` counts from the plan's first.  j is this
// thread's candidate; the results are in the threads it returns true for.
template <int LANES, bool PER_X0, int TEX, int ACC, class Tr>
__device__ __forceinline__ bool duo_rollout(const PlanParams &p, const Tr &tr, Duo<LANES> &sh, unsigned cta, int &j, float &J,
                                            float &margin, bool &feasible)
{
    const int lane = threadIdx.x & 31, c = lane / LANES, q = lane & (LANES - 1);
    const long long jl = (long long)cta * Duo<LANES>::kC + c;
    const bool live = jl < p.N;
    j = (int)jl;
    const bool geo = geometry_role(sh.flip);
    if (geo) duo_geometry<LANES, PER_X0, TEX>(p, tr, sh, j, q, c, live);
    else duo_forces<LANES, PER_X0, ACC>(p, tr, sh, j, q, c, live, J, margin, feasible);
    return live && !geo && q == 0;
}

}  // namespace atp
