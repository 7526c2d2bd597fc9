// est_kernel.cu - fused rollout, cost, lateral-acceleration margin and
// empirical argmin of the planar extended single-track (EST) model of arxiv
// 2603.20525 (App. "Extended Single-Track Vehicle Dynamics Model", Sec. IV-C),
// the formulation the paper sets beside the SRB model.
//
// One thread per candidate once the batch fills the GPU, two warps that share 32
// candidates below (the model has 7 states and one terrain lookup under the CoM
// per Euler step, plus four costmap lookups at the wheels when the terrain
// carries a costmap, reading Q17).  Pitch and roll are not states: they follow
// the terrain's normal under the CoM, whose components give their sines and
// cosines directly (1-2-3 convention), so the step needs two trigonometric
// evaluations (yaw and steering) and two arctangents (the virtual tires'
// slip).  The same FP32 conventions as the SRB kernel: explicit FMAs only,
// compensated sums for position, heading and velocity, positions relative to
// the terrain origin.  The reduction is the SRB kernel's fused tail.
#include <cuda_runtime.h>
#include <math_constants.h>

#include "duo.cuh"
#include "est_kernel.cuh"
#include "plan_tail.cuh"

namespace atp {

namespace {

// Bilinear lookup at (ox, oy) metres from the CoM; sets `off` for a query
// outside the map.
template <int TEX>
__device__ __forceinline__ float4 lookup(const Terrain &T, const Cell &cx, const Cell &cy, unsigned base, float ox,
                                         float oy, bool &off)
{
    float a, b;
    const float tx = axis(cx, fmaf(ox, T.inv_cell, cx.fc), a, off);
    const float ty = axis(cy, fmaf(oy, T.inv_cell, cy.fc), b, off);
    return bilerp<TEX>(T, cx, cy, base, tx, ty, a, b);
}

__device__ __forceinline__ float tire(const Veh &V, float Fz, float alpha)
{
    const float Ca = V.C * alpha;
    return Fz * (-Ca * V.mu) * rsq(fmaf(Ca, Ca, V.mu2));
}

template <bool PER_X0, int TEX>
__device__ __forceinline__ void est_one(const PlanParams &p, int j, float &J, float &margin, bool &feasible)
{
    const Veh &V = p.V;
    const Cost &Cc = p.C;
    const Terrain &T = p.T;
    // state x, y, psi, v_By, w_Bz, delta, v_Bx; x, y relative to the origin;
    // *_l the low parts of the compensated components
    float x, xl, y, yl, psi, psil = 0.f, vy, vyl = 0.f, wz, d, vx, vxl = 0.f;
    {
        float s[7];
        if (PER_X0) {
#pragma unroll
            for (int c = 0; c < 7; ++c) s[c] = p.x0_soa[(size_t)c * p.N + j];
        } else {
#pragma unroll
            for (int c = 0; c < 7; ++c) s[c] = p.x0[c];
        }
        two_sum(s[0], -T.x0_hi, x, xl);
        xl -= T.x0_lo;
        two_sum(s[1], -T.y0_hi, y, yl);
        yl -= T.y0_lo;
        psi = s[2]; vy = s[3]; wz = s[4]; d = s[5]; vx = s[6];
    }
    // wheel contact points in B (fl, fr, rl, rr): (+-L, +-e/2, -(h+R))
    bool done = false, off = false;
    const float h = p.h;
    const bool cm = T.has_cm != 0;
    double J64 = 0.0;
    float msm = CUDART_INF_F;      // smallest per-step margin so far and its control step
    int mstep = 0;
    // each interval's control is loaded one interval ahead, so the load's
    // latency overlaps the Euler steps
    float2 un = p.H > 0 ? __ldg(p.ctrl + j) : make_float2(0.f, 0.f);
    for (int k = 0; k < p.H; ++k) {
        const float2 u = un;
        if (k + 1 < p.H) un = __ldg(p.ctrl + (size_t)(k + 1) * p.N + j);
        const float dd = clamp_keep_nan(u.x, -V.ddmax, V.ddmax);
        const float ax = u.y;
        float sm = CUDART_INF_F;
        for (int sub = 0; sub < p.n_sub; ++sub) {
            if (done) continue;            // frozen at the goal
            const float gdx = (x - Cc.gx_hi) + (xl - Cc.gx_lo);
            const float gdy = (y - Cc.gy_hi) + (yl - Cc.gy_lo);
            if (fmaf(gdx, gdx, gdy * gdy) <= Cc.goal_r2) {
                done = true;
                continue;
            }
            // terrain under the CoM and its unit normal (reading Q1)
            const Cell cx = cell_of(x, xl, T.inv_cell, T.nx), cy = cell_of(y, yl, T.inv_cell, T.ny);
            const unsigned base = texel_base(cx, cy, T.nx);
            off = off || off_com(cx, cy);
            const float4 t = lookup<TEX>(T, cx, cy, base, 0.f, 0.f, off);
            const float rn = rsq(fmaf(t.y, t.y, fmaf(t.z, t.z, 1.f)));
            const float tx = -t.y * rn, ty = -t.z * rn, tz = rn;
            // 1-2-3 angles of the plane: sin(theta) = tau_x, cos(theta) =
            // |(tau_y, tau_z)|, sin(phi) = -tau_y / cos(theta), cos(phi) = tau_z / cos(theta)
            const float sth = tx;
            const float cth = sqrtf(fmaf(ty, ty, tz * tz));
            const float ict = rcp(cth);
            const float sph = -ty * ict, cph = tz * ict;
            float sps, cps, sd, cd;
            sincos_r(psi, sps, cps);
            sincos_r(d, sd, cd);
            // rotation body -> world (rows 0 and 1, and the third row's gravity)
            const float R00 = cth * cps, R01 = -cth * sps, R02 = sth;
            const float R10 = fmaf(cps * sph, sth, cph * sps);
            const float R11 = fmaf(-sph * sth, sps, cph * cps);
            const float R12 = -cth * sph;
            const float R21 = fmaf(cph * sth, sps, cps * sph);
            const float R22 = cph * cth;
            const float gBy = -V.g * R21, gBz = -V.g * R22;
            // virtual tires: normal forces with longitudinal load transfer, slip, force
            const float aBx = fmaf(-wz, vy, ax);
            const float Fzf = fmaf(-V.Kzzf, gBz, -V.Kzx * aBx);
            const float Fzr = fmaf(-V.Kzzr, gBz, V.Kzx * aBx);
            const float af = atan2_r(fmaf(wz, V.Lf, vy), vx) - d;
            const float ar = atan2_r(fmaf(-wz, V.Lr, vy), vx);
            const float Fyf = tire(V, Fzf, af);
            const float Fyr = tire(V, Fzr, ar);
            // A(xi) + B zeta
            const float dx = fmaf(R01, vy, R00 * vx);
            const float dy = fmaf(R11, vy, R10 * vx);
            const float dvy = fmaf(-wz, vx, fmaf(Fyf + Fyr, V.invM, gBy));
            const float dwz = fmaf(Fyf * V.Lf, cd, -Fyr * V.Lr) * V.invJzz;
            // lateral-acceleration constraint |a_By - g_By| < abar (Sec. IV-C)
            const float aBy = fmaf(wz, vx, dvy);
            const float m = V.abar - fabsf(aBy - gBy);
            margin = fminf(margin, m);
            sm = fminf(sm, m);
            // distance constraints: the costmap at the four contact points,
            // read only when the terrain has one (reading Q17)
            float csum = 0.f;
            if (cm) {
                const float ofx = fmaf(R02, -V.hR, R00 * V.Lf), ofy = fmaf(R12, -V.hR, R10 * V.Lf);
                const float orx = fmaf(R02, -V.hR, -R00 * V.Lr), ory = fmaf(R12, -V.hR, -R10 * V.Lr);
                const float lx = R01 * V.he, ly = R11 * V.he;
                const float cfl = lookup<TEX>(T, cx, cy, base, ofx + lx, ofy + ly, off).w;
                const float cfr = lookup<TEX>(T, cx, cy, base, ofx - lx, ofy - ly, off).w;
                const float crl = lookup<TEX>(T, cx, cy, base, orx + lx, ory + ly, off).w;
                const float crr = lookup<TEX>(T, cx, cy, base, orx - lx, ory - ly, off).w;
                csum = (cfl + cfr) + (crl + crr);
            }
            const float soft = fmaxf(fmaf(-m, Cc.inv_eps, 1.f), 0.f);
            const float L = fmaf(Cc.sigma * soft, soft, fmaf(Cc.wc * dd, dd, Cc.wt)) + csum;
            if (p.acc64) J64 += (double)(h * L);
            else J = fmaf(h, L, J);
            // forward Euler, steering angle clamped (reading Q5)
            acc2(x, xl, h * dx);
            acc2(y, yl, h * dy);
            acc2(psi, psil, h * wz);
            acc2(vy, vyl, h * dvy);
            wz = fmaf(h, dwz, wz);
            d = clamp_keep_nan(fmaf(h, dd, d), -V.dmax, V.dmax);
            acc2(vx, vxl, h * ax);
        }
        if (p.step_margin) p.step_margin[(size_t)k * p.N + j] = sm;
        if (sm < msm) {
            msm = sm;
            mstep = k;
        }
    }
    // final state: goal test and terminal cost Phi (Sec. IV-C)
    {
        const float gdx = (x - Cc.gx_hi) + (xl - Cc.gx_lo);
        const float gdy = (y - Cc.gy_hi) + (yl - Cc.gy_lo);
        const float d2 = fmaf(gdx, gdx, gdy * gdy);
        if (!done && d2 <= Cc.goal_r2) done = true;
        if (p.acc64) J = (float)(J64 + (double)(Cc.wg * sqrtf(d2)));
        else J = fmaf(Cc.wg, sqrtf(d2), J);
    }
    const float xs[7] = {(x + T.x0_hi) + (xl + T.x0_lo), (y + T.y0_hi) + (yl + T.y0_lo), psi + psil,
                         vy + vyl, wz, d, vx + vxl};
    bool finite = isfinite(J);
#pragma unroll
    for (int c = 0; c < 7; ++c) finite = finite && isfinite(xs[c]);
    if (!finite) J = CUDART_INF_F;
    feasible = finite && margin > 0.f;
    const uint8_t fl = (feasible ? ATP_FLAG_FEASIBLE : 0) | (done ? ATP_FLAG_DONE : 0) |
                       (off ? ATP_FLAG_OFFMAP : 0) | (finite ? 0 : ATP_FLAG_NONFINITE);
    if (p.cost) p.cost[j] = J;
    if (p.margin) p.margin[j] = margin;
    if (p.flags) p.flags[j] = fl;
    if (p.min_step) p.min_step[j] = mstep;
    if (p.xf) {
#pragma unroll
        for (int c = 0; c < 7; ++c) p.xf[(size_t)c * p.N + j] = xs[c];
    }
}

// ---- two warps per 32 candidates ---------------------------------------------
//
// As the SRB model's two-warp layouts (duo.cuh): position, yaw and steering of
// step t + 1 need the velocities of step t only, so one warp advances them and
// looks the terrain up while the other turns step t's plane into forces,
// velocities, margin and cost.  The expressions are est_one's, and so the bits.
struct EstDuo {
    float4 plane[2][32];      // gravity in B (y, z), cos(delta), delta
    float2 cost[2][32];       // costmap sum; done (0 or 1)
    float4 v[2][32];          // v_By, w_Bz, v_Bx
    float d2[32];             // final squared distance to the goal
    int flags[32];            // done, off the map, final state not finite
    int flip;
};

template <bool PER_X0, int TEX>
__device__ __forceinline__ void est_geometry(const PlanParams &p, EstDuo &sh, int j, int c, bool live)
{
    const Veh &V = p.V;
    const Cost &Cc = p.C;
    const Terrain &T = p.T;
    float x = 0.f, xl = 0.f, y = 0.f, yl = 0.f, psi = 0.f, psil = 0.f, d = 0.f;
    if (live) {
        const auto s = [&](int r) { return PER_X0 ? __ldg(p.x0_soa + (size_t)r * p.N + j) : p.x0[r]; };
        two_sum(s(0), -T.x0_hi, x, xl);
        xl -= T.x0_lo;
        two_sum(s(1), -T.y0_hi, y, yl);
        yl -= T.y0_lo;
        psi = s(2);
        d = s(5);
    }
    const float h = p.h;
    const bool cm = T.has_cm != 0;
    bool done = !live, off = false, offs = false, huge = false;
    float R00 = 0.f, R01 = 0.f, R10 = 0.f, R11 = 0.f;
    // the plane under the CoM, the rotation and the goal test, into buffer `par`
    const auto geometry = [&](int par, auto form) {
        const float gdx = (x - Cc.gx_hi) + (xl - Cc.gx_lo);
        const float gdy = (y - Cc.gy_hi) + (yl - Cc.gy_lo);
        done = done || fmaf(gdx, gdx, gdy * gdy) <= Cc.goal_r2;
        const Cell cx = cell_of(x, xl, T.inv_cell, T.nx), cy = cell_of(y, yl, T.inv_cell, T.ny);
        const unsigned base = texel_base(cx, cy, T.nx);
        offs = off_com(cx, cy);
        const float4 t = lookup<TEX>(T, cx, cy, base, 0.f, 0.f, offs);
        float sps, cps, sd, cd;
        sincos_g<decltype(form)::value>(psi, sps, cps);
        sincos_g<decltype(form)::value>(d, sd, cd);
        huge = fmaxf(fabsf(psi), fabsf(d)) >= kSincosMax;
        const float rn = rsq(fmaf(t.y, t.y, fmaf(t.z, t.z, 1.f)));
        const float tx = -t.y * rn, ty = -t.z * rn, tz = rn;
        const float sth = tx;
        const float cth = sqrtf(fmaf(ty, ty, tz * tz));
        const float ict = rcp(cth);
        const float sph = -ty * ict, cph = tz * ict;
        R00 = cth * cps;
        R01 = -cth * sps;
        const float R02 = sth;
        R10 = fmaf(cps * sph, sth, cph * sps);
        R11 = fmaf(-sph * sth, sps, cph * cps);
        const float R12 = -cth * sph;
        const float R21 = fmaf(cph * sth, sps, cps * sph);
        const float R22 = cph * cth;
        float csum = 0.f;
        if (cm) {
            const float ofx = fmaf(R02, -V.hR, R00 * V.Lf), ofy = fmaf(R12, -V.hR, R10 * V.Lf);
            const float orx = fmaf(R02, -V.hR, -R00 * V.Lr), ory = fmaf(R12, -V.hR, -R10 * V.Lr);
            const float lx = R01 * V.he, ly = R11 * V.he;
            const float cfl = lookup<TEX>(T, cx, cy, base, ofx + lx, ofy + ly, offs).w;
            const float cfr = lookup<TEX>(T, cx, cy, base, ofx - lx, ofy - ly, offs).w;
            const float crl = lookup<TEX>(T, cx, cy, base, orx + lx, ory + ly, offs).w;
            const float crr = lookup<TEX>(T, cx, cy, base, orx - lx, ory - ly, offs).w;
            csum = (cfl + cfr) + (crl + crr);
        }
        sh.plane[par][c] = make_float4(-V.g * R21, -V.g * R22, cd, d);
        sh.cost[par][c] = make_float2(csum, done ? 1.f : 0.f);
    };
    const auto advance = [&](int par) {
        geometry(par, Fast{});
        if (__any_sync(kFull, huge)) geometry(par, Slow{});
    };
    advance(0);
    pair_barrier();
    int par = 0;
    float un = live ? __ldg(&p.ctrl[j].x) : 0.f;
    for (int k = 0; k < p.H; ++k) {
        const float dd = clamp_keep_nan(un, -V.ddmax, V.ddmax);
        if (live && k + 1 < p.H) un = __ldg(&p.ctrl[(size_t)(k + 1) * p.N + j].x);
        const bool idle = __all_sync(kFull, done);     // every candidate frozen at the goal
        for (int sub = 0; sub < p.n_sub; ++sub) {
            if (!idle) {
                const float4 v = sh.v[par][c];
                const float vy = v.x, wz = v.y, vx = v.z;
                const bool go = !done;
                off = off || (go && offs);
                const float dx = fmaf(R01, vy, R00 * vx);
                const float dy = fmaf(R11, vy, R10 * vx);
                float nx = x, nxl = xl, ny = y, nyl = yl, np_ = psi, npl = psil;
                acc2(nx, nxl, h * dx);
                acc2(ny, nyl, h * dy);
                acc2(np_, npl, h * wz);
                const float nd = clamp_keep_nan(fmaf(h, dd, d), -V.dmax, V.dmax);
                x = sel(go, nx, x); xl = sel(go, nxl, xl); y = sel(go, ny, y); yl = sel(go, nyl, yl);
                psi = sel(go, np_, psi); psil = sel(go, npl, psil); d = sel(go, nd, d);
                advance(par ^ 1);
            }
            pair_barrier();
            par ^= 1;
        }
    }
    const float gdx = (x - Cc.gx_hi) + (xl - Cc.gx_lo);
    const float gdy = (y - Cc.gy_hi) + (yl - Cc.gy_lo);
    const float xs[4] = {(x + T.x0_hi) + (xl + T.x0_lo), (y + T.y0_hi) + (yl + T.y0_lo), psi + psil, d};
    const bool finite = isfinite(xs[0]) && isfinite(xs[1]) && isfinite(xs[2]) && isfinite(xs[3]);
    sh.d2[c] = fmaf(gdx, gdx, gdy * gdy);
    sh.flags[c] = (done ? ATP_FLAG_DONE : 0) | (off ? ATP_FLAG_OFFMAP : 0) | (finite ? 0 : ATP_FLAG_NONFINITE);
    if (live && p.xf) {
        const size_t N = (size_t)p.N;
        p.xf[j] = xs[0];
        p.xf[N + j] = xs[1];
        p.xf[2 * N + j] = xs[2];
        p.xf[5 * N + j] = xs[3];
    }
    pair_barrier();
}

template <bool PER_X0>
__device__ __forceinline__ void est_forces(const PlanParams &p, EstDuo &sh, int j, int c, bool live, float &J,
                                           float &margin, bool &feasible)
{
    const Veh &V = p.V;
    const Cost &Cc = p.C;
    float vy = 0.f, vyl = 0.f, wz = 0.f, vx = 0.f, vxl = 0.f;
    if (live) {
        const auto s = [&](int r) { return PER_X0 ? __ldg(p.x0_soa + (size_t)r * p.N + j) : p.x0[r]; };
        vy = s(3);
        wz = s(4);
        vx = s(6);
    }
    const float h = p.h;
    double J64 = 0.0;
    float msm = CUDART_INF_F;
    int mstep = 0;
    sh.v[0][c] = make_float4(vy, wz, vx, 0.f);
    pair_barrier();
    int par = 0;
    bool idle = false;
    float2 un = live ? __ldg(p.ctrl + j) : make_float2(0.f, 0.f);
    for (int k = 0; k < p.H; ++k) {
        const float dd = clamp_keep_nan(un.x, -V.ddmax, V.ddmax), ax = un.y;
        if (live && k + 1 < p.H) un = __ldg(p.ctrl + (size_t)(k + 1) * p.N + j);
        idle = idle || __all_sync(kFull, sh.cost[par][c].y != 0.f);    // for good: the buffers stay as they are
        float sm = CUDART_INF_F;
        for (int sub = 0; sub < p.n_sub; ++sub) {
            if (!idle) {
                const float4 g = sh.plane[par][c];
                const float2 cd2 = sh.cost[par][c];
                const float gBy = g.x, gBz = g.y, cd = g.z, d = g.w, csum = cd2.x;
                const bool go = cd2.y == 0.f;
                // virtual tires: normal forces with longitudinal load transfer, slip, force
                const float aBx = fmaf(-wz, vy, ax);
                const float Fzf = fmaf(-V.Kzzf, gBz, -V.Kzx * aBx);
                const float Fzr = fmaf(-V.Kzzr, gBz, V.Kzx * aBx);
                const float af = atan2_r(fmaf(wz, V.Lf, vy), vx) - d;
                const float ar = atan2_r(fmaf(-wz, V.Lr, vy), vx);
                const float Fyf = tire(V, Fzf, af);
                const float Fyr = tire(V, Fzr, ar);
                const float dvy = fmaf(-wz, vx, fmaf(Fyf + Fyr, V.invM, gBy));
                const float dwz = fmaf(Fyf * V.Lf, cd, -Fyr * V.Lr) * V.invJzz;
                // lateral-acceleration constraint |a_By - g_By| < abar (Sec. IV-C)
                const float aBy = fmaf(wz, vx, dvy);
                const float m = V.abar - fabsf(aBy - gBy);
                float nvy = vy, nvyl = vyl, nvx = vx, nvxl = vxl;
                acc2(nvy, nvyl, h * dvy);
                const float nwz = fmaf(h, dwz, wz);
                acc2(nvx, nvxl, h * ax);
                vy = sel(go, nvy, vy); vyl = sel(go, nvyl, vyl); wz = sel(go, nwz, wz);
                vx = sel(go, nvx, vx); vxl = sel(go, nvxl, vxl);
                sh.v[par ^ 1][c] = make_float4(vy, wz, vx, 0.f);
                margin = sel(go, fminf(margin, m), margin);
                sm = sel(go, fminf(sm, m), sm);
                const float soft = fmaxf(fmaf(-m, Cc.inv_eps, 1.f), 0.f);
                const float L = fmaf(Cc.sigma * soft, soft, fmaf(Cc.wc * dd, dd, Cc.wt)) + csum;
                if (p.acc64) J64 += go ? (double)(h * L) : 0.0;
                else J = sel(go, fmaf(h, L, J), J);
            }
            pair_barrier();
            par ^= 1;
        }
        if (live && p.step_margin) p.step_margin[(size_t)k * p.N + j] = sm;
        if (sm < msm) {
            msm = sm;
            mstep = k;
        }
    }
    pair_barrier();                       // the geometry warp's final state is stored
    if (!live) return;
    const float d2 = sh.d2[c];
    if (p.acc64) J = (float)(J64 + (double)(Cc.wg * sqrtf(d2)));
    else J = fmaf(Cc.wg, sqrtf(d2), J);
    const float xs[3] = {vy + vyl, wz, vx + vxl};
    const int gfl = sh.flags[c];
    const bool finite = isfinite(J) && !(gfl & ATP_FLAG_NONFINITE) && isfinite(xs[0]) && isfinite(xs[1]) && isfinite(xs[2]);
    if (!finite) J = CUDART_INF_F;
    feasible = finite && margin > 0.f;
    if (p.cost) p.cost[j] = J;
    if (p.margin) p.margin[j] = margin;
    if (p.flags)
        p.flags[j] = (feasible ? ATP_FLAG_FEASIBLE : 0) | (gfl & (ATP_FLAG_DONE | ATP_FLAG_OFFMAP)) |
                     (finite ? 0 : ATP_FLAG_NONFINITE);
    if (p.min_step) p.min_step[j] = mstep;
    if (p.xf) {
        const size_t N = (size_t)p.N;
        p.xf[3 * N + j] = xs[0];
        p.xf[4 * N + j] = xs[1];
        p.xf[6 * N + j] = xs[2];
    }
}

template <bool PER_X0, int TEX>
__global__ void __launch_bounds__(kPlanBlock) est_duo_kernel(const __grid_constant__ PlanParams p)
{
    __shared__ EstDuo sh;
    const int c = threadIdx.x & 31, j = blockIdx.x * 32 + c;
    const bool live = j < p.N;
    float J = 0.f, margin = CUDART_INF_F;
    bool feasible = false;
    const bool geo = geometry_role(sh.flip);
    if (geo) est_geometry<PER_X0, TEX>(p, sh, j, c, live);
    else est_forces<PER_X0>(p, sh, j, c, live, J, margin, feasible);
    plan_tail(p, j, live && !geo, J, feasible, gridDim.x);
}

// Candidates up to which two warps share 32: 152 x 10 x 32, where the two meet
// (scaled workload at H = 50, us per plan, two warps / one thread: 79 / 121 at
// 2048 candidates, 85 / 122 at 16384, 107 / 132 at 32768, 148 / 147 at 49152,
// 181 / 178 at 65536; with a costmap 170 / 243 at 16384, 243 / 254 at 49152).
constexpr int kEstDuoMaxN = 48640;

template <bool PER_X0, int TEX>
__global__ void __launch_bounds__(kPlanBlock) est_kernel(const __grid_constant__ PlanParams p)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    const bool live = j < p.N;
    float J = 0.f, margin = CUDART_INF_F;
    bool feasible = false;
    if (live) est_one<PER_X0, TEX>(p, j, J, margin, feasible);
    plan_tail(p, j, live, J, feasible, gridDim.x);
}

template <int TEX>
cudaError_t launch_tex(const PlanParams &p, cudaStream_t stream)
{
    const bool per = p.x0_soa != nullptr;
    if (p.N <= kEstDuoMaxN) {
        const dim3 grid((unsigned)((p.N + 31) / 32));
        if (per) est_duo_kernel<true, TEX><<<grid, kPlanBlock, 0, stream>>>(p);
        else est_duo_kernel<false, TEX><<<grid, kPlanBlock, 0, stream>>>(p);
    } else {
        const dim3 grid((unsigned)(((size_t)p.N + kPlanBlock - 1) / kPlanBlock));
        if (per) est_kernel<true, TEX><<<grid, kPlanBlock, 0, stream>>>(p);
        else est_kernel<false, TEX><<<grid, kPlanBlock, 0, stream>>>(p);
    }
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_est(const PlanParams &p, cudaStream_t stream)
{
    return p.tex_format == TEX_F32 ? launch_tex<TEX_F32>(p, stream) : launch_tex<TEX_BF16>(p, stream);
}

}  // namespace atp
