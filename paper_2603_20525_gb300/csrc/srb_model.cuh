// srb_model.cuh - FP32 device model of the single-rigid-body (SRB) off-road
// vehicle of arxiv 2603.20525, Sec. IV-A, with the sigmoid tire of Sec. III-A,
// the energy stability margin of Sec. IV-B and the running cost of Sec. IV-C.
//
// A candidate's state lives in registers for the whole horizon (in one
// thread, or repeated in the two or four threads that share its wheels), so a
// rollout step reads memory only for the four bilinear terrain lookups (16
// texels).  A wheel is written as its geometry (what depends on position and
// attitude: the lookup, the slope normal, the extension) and its forces
// (what depends on the velocities).
//
// Precision.  The arithmetic is FP32, compiled without implicit FMA
// contraction: every fused multiply-add is written as fmaf (or as fma2, its
// packed two-wide form, which rounds each half the same way), so the rounding
// of each expression is fixed by the source and the same in every kernel that
// inlines it.  The slowly varying, large-magnitude
// state components (position, heading and linear velocity) are accumulated as
// unevaluated sums hi + lo of two floats (Kahan's compensated summation per
// step, Knuth's TwoSum where the start is taken into the terrain frame), and
// positions are
// kept relative to the terrain origin and split into an integer cell and a
// fraction before the lookup.  Without that, the rounding of a 20-100 m
// coordinate (1e-6 m per Euler step) walks the wheels across the terrain by
// ~1e-5 m over a horizon, which the spring turns into force errors far above
// the 1e-4 relative agreement with the FP64 oracle.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "fastmath.cuh"

namespace atp {

// Vehicle constants in FP32, derived on the host in FP64 (App. B notation).
struct Veh {
    float M, halfM, invM;
    float dJyz, dJxz, dJxy;          // Jyy-Jzz, Jxx-Jzz, Jxx-Jyy
    float invJxx, invJyy, invJzz;
    float Lf, Lr, he, hR;            // he = e / 2
    float kf, kr, bf, br;
    float Fsf, Fsr;                  // nominal tire loading (g/2) K_zz,i
    float C, mu, mu2;
    float dmax, ddmax, g;
    float MgRbar;                    // M g Rbar
    float cpb, spb;                  // cos(phibar), sin(phibar)
    float tip;                       // pi/2 - phibar: roll at which U_ESM = 0
    // planar (EST) model: load-transfer coefficients and the critical lateral
    // acceleration M g / (2 K_zy)
    float Kzzf, Kzzr, Kzx, abar;
};

struct Cost {
    float wt, wc, wg, sigma, inv_eps;
    float gx_hi, gx_lo, gy_hi, gy_lo;  // goal relative to the terrain origin
    float goal_r2;
};

// Texel formats (ATP_TERRAIN_*): F32 = float4 (f, f_x, f_y, cost) per node;
// BF16 = four bf16 per node (f - plane, f_x - plane_x, f_y - plane_y, cost)
// with the FP32 plane (c0, cx, cy) of the node's 8 x 8 block.  F32W is F32
// with a window of the texels staged in the CTA's shared memory (`atp_win`,
// ww x wh nodes from node (wx0, wy0)): a lookup whose four corners lie in
// the window reads them there, any other from global memory.
enum { TEX_F32 = 0, TEX_BF16 = 1, TEX_F32W = 2 };

// the staged window of TEX_F32W (dynamic shared memory of the staging kernel)
extern __shared__ float4 atp_win[];

struct Terrain {
    const float4 *tex;               // F32 texels, row-major
    const uint2 *tex16;              // BF16 texels, row-major
    const float4 *plane16;           // BF16 block planes [ceil(ny/8)][ceil(nx/8)]
    int nbx;                         // blocks per row
    int nx, ny;
    int has_cm;                      // the texels carry a costmap
    float inv_cell;                  // 1 / cell
    float x0_hi, x0_lo, y0_hi, y0_lo;  // terrain origin
    int wx0, wy0, ww, wh;            // TEX_F32W: the staged window (ww, wh >= 2)
};

// x + y = s + e exactly (Knuth's TwoSum; no ordering precondition).
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// hi + lo += d, with the carried low part folded into the increment first
// (Kahan's compensated summation; the new low part by Dekker's Fast2Sum,
// exact while |hi| >= |d + lo|, which holds for a state component and its
// increment over one Euler step except near the component's zero, where
// the plain FP32 sum it reduces to is accurate to the component's own small
// magnitude).  Folding keeps hi the FP32 value nearest the compensated sum,
// so the dynamics, which read hi alone, see the state as exactly
// accumulated; a low part summed on its own instead leaves hi the plain FP32
// running sum, whose error grows with every step (a constant increment
// rounds the same way each time).
__device__ __forceinline__ void acc2(float &hi, float &lo, float d)
{
    const float y = __fadd_rn(d, lo);
    const float s = __fadd_rn(hi, y);
    lo = __fsub_rn(y, __fsub_rn(s, hi));
    hi = s;
}

// Energy stability margin (Sec. IV-B): U = +/- M g Rbar (1 - sin(|phi| +
// phibar)) cos(theta), positive while the CoM is inside the footprint,
// |phi| < pi/2 - phibar.  sin(|phi| + phibar) is expanded with the already
// computed sin(phi), cos(phi), so it costs no extra transcendental.
__device__ __forceinline__ float esm(const Veh &V, float ph, float sph, float cph, float cth)
{
    float sabs = ph < 0.f ? -sph : sph;                  // sin(|phi|)
    float s = fmaf(sabs, V.cpb, cph * V.spb);            // sin(|phi| + phibar)
    float u = V.MgRbar * (1.f - s) * cth;
    return fabsf(ph) < V.tip ? u : -u;
}

// 1.5 x 2^23: adding it to |u| <= 2^22 rounds u to a whole number in the low
// mantissa bits, at FADD latency instead of a conversion's (F2I, I2F and FRND
// run at a quarter rate and about five times the latency).
constexpr float kMagic = 12582912.f;
constexpr unsigned kMagicBits = 0x4b400000u;
constexpr float kMaxCell = 2097152.f;        // 2^21: the CoM's cell is clamped to +-2^21

// One axis of the CoM in cell units: the fraction fc of its cell, and the map
// as seen from that cell: its first node lo, its last node hi (whole numbers,
// exact), the last lookup cell in magic form (kMagic + n - 2 - cell), and the
// cell itself in magic form.
struct Cell {
    float fc, lo, hi, tmax, t;
};

// From the compensated coordinate hi + lo (metres from the origin).  A NaN
// takes the low edge.  WRAP: a position 2^31 cells or more beyond the map (a
// rollout that has diverged) takes the opposite edge's texels, as the plans'
// saturating 32-bit cell sums always have; it is off the map either way.
template <bool WRAP = true>
__device__ __forceinline__ Cell cell_of(float hi, float lo, float inv_cell, int n)
{
    Cell c;
    const float u = fminf(fmaxf(hi * inv_cell, -kMaxCell), kMaxCell);   // NaN -> low edge
    c.t = __fadd_rd(u, kMagic);
    const float fl = c.t - kMagic;                                      // floor(u)
    const float f = fmaf(lo, inv_cell, fmaf(hi, inv_cell, -fl));
    c.fc = !WRAP || fabsf(f) < 2143289344.f ? f : -f;                   // 2^31 - 2^22
    c.lo = -fl;
    c.hi = (float)(n - 1) - fl;
    c.tmax = (kMagic + (float)(n - 2)) - fl;
    return c;
}

// One axis of a lookup at `u` cells from the CoM's cell: returns the lookup
// cell in [0, n-2] (in magic form) and the weight w in [0, 1] (queries clamped
// to the map, reading Q10), and sets `off` for a query outside the map.  Only
// min, max and additions: the clamp of the coordinate gives the weights 0 and
// 1 beyond the map, and the coordinate differs from its clamp exactly when the
// query is off the map.  A NaN takes the low edge and does not set `off` (the
// caller's off_com does when the position itself is NaN); every index lies on
// the map whatever u is.
__device__ __forceinline__ float axis(const Cell &c, float u, float &w, bool &off)
{
    const float uc = fminf(fmaxf(u, c.lo), c.hi);
    const float t = fminf(__fadd_rd(uc, kMagic), c.tmax);
    w = uc - (t - kMagic);
    off = off || u < uc || u > uc;
    return t;
}

// the CoM is so far below the map's edge, or NaN, that its cell was clamped
__device__ __forceinline__ bool off_com(const Cell &cx, const Cell &cy)
{
    return cx.lo >= kMaxCell || cy.lo >= kMaxCell;
}

// texel index of the CoM's cell less the magic bits of a lookup's two axes:
// texel_index(base, tx, ty, nx) = j nx + i, modulo 2^32 (a map has at most
// 2^32 nodes)
__device__ __forceinline__ unsigned texel_base(const Cell &cx, const Cell &cy, int nx)
{
    return (__float_as_uint(cy.t) - 2u * kMagicBits) * (unsigned)nx + (__float_as_uint(cx.t) - 2u * kMagicBits);
}
__device__ __forceinline__ unsigned texel_index(unsigned base, float tx, float ty, int nx)
{
    return __float_as_uint(ty) * (unsigned)nx + (__float_as_uint(tx) + base);
}
// the lookup cell along one axis
__device__ __forceinline__ int cell_index(const Cell &c, float t)
{
    return (int)(__float_as_uint(t) + __float_as_uint(c.t) - 2u * kMagicBits);
}

__device__ __forceinline__ float lerp2d(float t00, float t10, float t01, float t11, float a, float b)
{
    const float lo = fmaf(a, t10 - t00, t00), hi = fmaf(a, t11 - t01, t01);
    return fmaf(b, hi - lo, lo);
}

// lerp2d on two channels at once, bit for bit the same
__device__ __forceinline__ float2 lerp2d2(float2 t00, float2 t10, float2 t01, float2 t11, float2 a,
                                          float2 b)
{
    const float2 lo = fma2(a, sub2(t10, t00), t00), hi = fma2(a, sub2(t11, t01), t01);
    return fma2(b, sub2(hi, lo), lo);
}

// bilinear height, slopes and (when the terrain has a costmap) cost
__device__ __forceinline__ float4 lerp4(float4 t00, float4 t10, float4 t01, float4 t11, float a, float b,
                                        bool cm)
{
    const float2 a2 = splat2(a), b2 = splat2(b);
    const float2 xy = lerp2d2(make_float2(t00.x, t00.y), make_float2(t10.x, t10.y),
                              make_float2(t01.x, t01.y), make_float2(t11.x, t11.y), a2, b2);
    const float2 zw = lerp2d2(make_float2(t00.z, t00.w), make_float2(t10.z, t10.w),
                              make_float2(t01.z, t01.w), make_float2(t11.z, t11.w), a2, b2);
    return make_float4(xy.x, xy.y, zw.x, cm ? zw.y : 0.f);
}

// height of a block's plane (c0, cx, cy) at node (i, j): c0 + cx (i mod 8) +
// cy (j mod 8), every operation rounded on its own
__device__ __forceinline__ float block_plane(float4 P, int i, int j)
{
    return __fadd_rn(__fadd_rn(P.x, __fmul_rn(P.y, (float)(i & 7))), __fmul_rn(P.z, (float)(j & 7)));
}

// one BF16 texel decoded from its block's plane, at (x, y) within the block:
// height = block plane + residual
__device__ __forceinline__ float4 texel16(const Terrain &T, uint2 u, float4 P, float x, float y)
{
    float4 t;
    t.x = __fadd_rn(__fadd_rn(__fadd_rn(P.x, __fmul_rn(P.y, x)), __fmul_rn(P.z, y)), __uint_as_float(u.x << 16));
    t.y = __fadd_rn(__fmul_rn(P.y, T.inv_cell), __uint_as_float(u.x & 0xffff0000u));
    t.z = __fadd_rn(__fmul_rn(P.z, T.inv_cell), __uint_as_float(u.y << 16));
    t.w = __uint_as_float(u.y & 0xffff0000u);
    return t;
}

// v mod 8 as a float, by its bits
__device__ __forceinline__ float mod8(int v) { return __uint_as_float(0x4b000000u | (unsigned)(v & 7)) - 8388608.f; }

// Bilinear lookup on BF16 texels.  The four corners mostly share one block, but
// loading the other planes only in the lanes that straddle an edge was slower
// (branches on the lookup's chain).
__device__ __forceinline__ float4 bilerp16(const Terrain &T, int i, int j, float a, float b, bool cm)
{
    const uint2 *r0 = T.tex16 + (size_t)j * T.nx + i, *r1 = r0 + T.nx;
    const uint2 u00 = __ldg(r0), u10 = __ldg(r0 + 1), u01 = __ldg(r1), u11 = __ldg(r1 + 1);
    const float4 *P = T.plane16 + (size_t)(j >> 3) * T.nbx + (i >> 3);
    const int ex = ((i & 7) + 1) >> 3, ey = ((j & 7) + 1) >> 3 ? T.nbx : 0;
    const float4 P00 = __ldg(P), P10 = __ldg(P + ex), P01 = __ldg(P + ey), P11 = __ldg(P + ex + ey);
    const float x0 = mod8(i), x1 = mod8(i + 1), y0 = mod8(j), y1 = mod8(j + 1);
    return lerp4(texel16(T, u00, P00, x0, y0), texel16(T, u10, P10, x1, y0), texel16(T, u01, P01, x0, y1),
                 texel16(T, u11, P11, x1, y1), a, b, cm);
}

// The lookup at cell (tx, ty) (magic form) with weights (a, b), seen from the
// CoM's cell (cx, cy) whose texel_base is `base`.
template <int TEX>
__device__ __forceinline__ float4 bilerp(const Terrain &T, const Cell &cx, const Cell &cy, unsigned base, float tx,
                                         float ty, float a, float b)
{
    const bool cm = T.has_cm != 0;
    if (TEX == TEX_F32) {
        const unsigned o = texel_index(base, tx, ty, T.nx);
        const float4 *r0 = T.tex + o, *r1 = T.tex + (size_t)(o + (unsigned)T.nx);
        return lerp4(__ldg(r0), __ldg(r0 + 1), __ldg(r1), __ldg(r1 + 1), a, b, cm);
    } else if (TEX == TEX_F32W) {
        // one generic pointer into the window or the texel array, so that a
        // warp whose lookups fall on both sides still issues four loads
        const int i = cell_index(cx, tx), j = cell_index(cy, ty);
        const unsigned li = (unsigned)(i - T.wx0), lj = (unsigned)(j - T.wy0);
        const bool in = li < (unsigned)(T.ww - 1) && lj < (unsigned)(T.wh - 1);
        const float4 *r0 = in ? atp_win + (lj * (unsigned)T.ww + li) : T.tex + (size_t)j * T.nx + i;
        const int s = in ? T.ww : T.nx;
        return lerp4(r0[0], r0[1], r0[s], r0[s + 1], a, b, cm);
    } else {
        return bilerp16(T, cell_index(cx, tx), cell_index(cy, ty), a, b, cm);
    }
}

// What the force of one wheel needs from the state's position and attitude
// alone: the local slope-normal tau in B (and 1 / tau_z) and the suspension
// extension chi at the contact point, and the costmap there.
struct WheelGeo {
    float tx, ty, tz, itz, chi, cost;
};

// What the lookup at one wheel gives: the interpolated slopes, the CoM height
// above the terrain there P_z - f (with the compensated CoM height), the
// costmap.
struct WheelGround {
    float fx, fy, Q, cost;
};

// One wheel's ground (Sec. IV-A): contact point P = p + R rho and the terrain
// below it.  cx, cy is the CoM's cell and z_hi + z_lo its height.
template <int TEX>
__device__ __forceinline__ WheelGround wheel_ground(const Veh &V, const Terrain &T, const float R[9], const Cell &cx,
                                                    const Cell &cy, unsigned base, float z_hi, float z_lo, float rx,
                                                    float ry, bool &off)
{
    // offset of the contact point from the CoM in W: R (rx, ry, -(h+R))
    const float2 oxy = fma2(splat2(rx), make_float2(R[0], R[3]),
                            fma2(splat2(ry), make_float2(R[1], R[4]),
                                 make_float2(-V.hR * R[2], -V.hR * R[5])));
    const float oz = fmaf(rx, R[6], fmaf(ry, R[7], -V.hR * R[8]));
    // terrain below the contact point
    const float2 u = fma2(oxy, splat2(T.inv_cell), make_float2(cx.fc, cy.fc));
    float a, bb;
    const float tx = axis(cx, u.x, a, off), ty = axis(cy, u.y, bb, off);
    const float4 t = bilerp<TEX>(T, cx, cy, base, tx, ty, a, bb);
    return {t.y, t.z, (z_hi - t.x) + (oz + z_lo), t.w};
}

// The slope-normal tau ~ (-f_x, -f_y, 1) (reading Q1) resolved in B and the
// extension chi along it.
__device__ __forceinline__ WheelGeo wheel_geo(const float R[9], const WheelGround &t)
{
    // tau in B = R^T (-f_x, -f_y, 1)
    const float2 txy = fma2(make_float2(-R[3], -R[4]), splat2(t.fy),
                            fma2(make_float2(-R[0], -R[1]), splat2(t.fx), make_float2(R[6], R[7])));
    WheelGeo g;
    g.tx = txy.x;
    g.ty = txy.y;
    g.tz = fmaf(-R[5], t.fy, fmaf(-R[2], t.fx, R[8]));
    g.itz = rcp(g.tz);
    g.chi = t.Q * g.itz;
    g.cost = t.cost;
    return g;
}

// 3-2-1 rotation, body -> world (Sec. IV-A)
__device__ __forceinline__ void rotation(float sps, float cps, float sth, float cth, float sph, float cph, float R[9])
{
    R[0] = cps * cth;
    R[1] = fmaf(cps * sph, sth, -cph * sps);
    R[2] = fmaf(cph * cps, sth, sph * sps);
    R[3] = cth * sps;
    R[4] = fmaf(sph * sps, sth, cph * cps);
    R[5] = fmaf(cph * sps, sth, -cps * sph);
    R[6] = -sth;
    R[7] = cth * sph;
    R[8] = cph * cth;
}

// What one wheel contributes to the force and moment sums.
struct WheelOut {
    float Fz, Fy, cost;
};

// One wheel's forces (Sec. IV-A) at the body velocity (vx, vy, vz) and rate
// (wx, wy, wz): the contact point's body velocity v + w x rho, the extension
// rate chi_dot, spring and damper with liftoff, slip angle and sigmoid tire
// force.  PAIRED takes the extension rate's inner pair as a packed pair (the
// same bits).  RATIO forms F_y as F_z (F_y / F_z), the adjoint's order, instead
// of multiplying from the left.
template <bool PAIRED = false, bool RATIO = false>
__device__ __forceinline__ WheelOut wheel_dyn(const Veh &V, const WheelGeo &g, float vx, float vy, float vz,
                                              float wx, float wy, float wz, float rx, float ry, float k,
                                              float b, float Fs, float di)
{
    // body velocity of the contact point: v + w x rho
    const float vix = fmaf(-wz, ry, fmaf(-wy, V.hR, vx));
    const float viy = fmaf(wx, V.hR, fmaf(wz, rx, vy));
    const float viz = fmaf(-wy, rx, fmaf(wx, ry, vz));
    // omega x b_z in B is (w_y, -w_x, 0)
    float chid;
    if constexpr (PAIRED) {
        const float2 rel = fma2(splat2(g.chi), make_float2(wx, -wy), make_float2(viy, vix));
        chid = fmaf(g.tz, viz, fmaf(g.ty, rel.x, g.tx * rel.y)) * g.itz;
    } else {
        chid = fmaf(g.tz, viz, fmaf(g.ty, fmaf(g.chi, wx, viy), g.tx * fmaf(-g.chi, wy, vix))) * g.itz;
    }
    const float Fk = fmaxf(fmaf(-k, g.chi, Fs), 0.f);
    const float Fz = Fk > 0.f ? fmaxf(fmaf(-b, chid, Fk), 0.f) : 0.f;   // = F_k + max(-b chid, -F_k)
    const float alpha = atan2_r(viy, vix) - di;
    const float Ca = V.C * alpha;
    const float is = rsq(fmaf(Ca, Ca, V.mu2));
    const float Fy = RATIO ? Fz * ((-Ca * V.mu) * is) : Fz * (-Ca * V.mu) * is;
    WheelOut w;
    w.Fz = Fz;
    w.Fy = Fy;
    w.cost = g.cost;
    return w;
}

// Per-step body quantities the four wheels share.
struct Body {
    float R[9];
    Cell cx, cy;             // CoM cell
    unsigned base;           // its texel_base
    float z_hi, z_lo;        // CoM height
    float vx, vy, vz, wx, wy, wz;
};

// One wheel (Sec. IV-A): its geometry, then its forces at the body's
// velocities.
template <int TEX>
__device__ __forceinline__ WheelOut wheel(const Veh &V, const Terrain &T, const Body &B, float rx, float ry,
                                          float k, float b, float Fs, float di, bool &off)
{
    const WheelGeo g =
        wheel_geo(B.R, wheel_ground<TEX>(V, T, B.R, B.cx, B.cy, B.base, B.z_hi, B.z_lo, rx, ry, off));
    return wheel_dyn(V, g, B.vx, B.vy, B.vz, B.wx, B.wy, B.wz, rx, ry, k, b, Fs, di);
}

}  // namespace atp
