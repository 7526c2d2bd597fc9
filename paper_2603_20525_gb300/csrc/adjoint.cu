// adjoint.cu - hand-written reverse-mode adjoint of the discrete rollout
// (arxiv 2603.20525, Sec. IV-A..IV-C): the gradient, with respect to the raw
// control sequence u of each of K candidates, of its cost J = sum over Euler
// steps of h L + Phi, or of its ESM margin, the minimum of U_ESM over every
// state of the trajectory (Sec. IV-B; the constraint the soft cost guards).
// The margin's gradient is that of U_ESM at the state holding the minimum
// (the first one on ties), as a subgradient of the minimum.
//
// Two kernels.  The forward one is the two-warp rollout (duo.cuh), which also
// writes every Euler step's start state.  Given those states, the steps'
// derivatives do not depend on one another, only their product with the
// adjoint does: in the backward kernel each lane of a candidate's warps
// linearises one Euler step (the 13 x 13 matrix by which the step's adjoint
// changes, column by column into shared memory), and then one warp runs the
// recursion lam <- lam + M lam + c over those steps, one column per lane.
// The recursion's step is one round trip through shared memory and 13 FMAs,
// instead of the step's whole forward and reverse arithmetic on the serial
// chain.  Walking the steps back with their arithmetic on the chain, beside a
// recomputation from checkpoints, took (ms) 0.73 for 64 candidates of 400
// steps, 0.78 for 4096 of 300, 1.28 and 2.62 for 16384 of 200 and 400, 4.16 for
// 32768 of 400 and 7.46 for 131072 of 200; this way they take 0.21, 0.43, 0.95,
// 1.85, 3.86 and 6.91.  The forward chain bounds the first (about 0.15), the
// linearisation's issue and the seven warps per SM that its shared memory holds
// the others.
//
// Linearising a step differentiates the Euler update, the state derivative
// A(xi) + B zeta, the force and moment sums, every wheel (contact kinematics,
// bilinear terrain, suspension with liftoff, slip and tire), the rotation and
// the running cost with its ESM soft constraint.  Branches (spring and damper
// liftoff, steering clamps, off-map clamping, the goal test) follow the
// forward pass's choice, so the result is the derivative of the
// piecewise-smooth discrete map along the primal trajectory.
#include <cuda_runtime.h>
#include <math_constants.h>

#include <algorithm>

#include "adjoint.cuh"
#include "duo.cuh"

namespace atp {

namespace {

// ---- linearisation of one Euler step ---------------------------------------

// Rows of the step's matrix, the components of the adjoint after the step.
enum { X, Y, Z, PSI, TH, PH, VX, VY, VZ, WX, WY, WZ, DE, kRows };
// Columns: the same components before the step, then the two gradients.
constexpr int kGdd = 13, kGax = 14, kCols = 15;
// One column: the 13 rows, the constant c, (in column kGdd) whether the
// steering rate is inside its limit, and the component's own factor: 1, or 0
// for a steering angle at its clamp.
constexpr int kColFloats = 16;
// floats per step, padded so that the lanes' 16-byte stores fall on distinct banks
constexpr int kStepFloats = kCols * kColFloats + 4;

// gradients of one wheel's F_z: x, y, z, psi, theta, phi, v, w
struct WheelGrad {
    float Fz, Fy;            // the forces
    float ratio;             // F_y / F_z
    float g[12];             // dF_z
    float a[5], ad;          // F_z d(F_y / F_z) / d(vx, vy, wx, wy, wz) and / d(delta)
    float c[6];              // costmap rate: x, y, (z), psi, theta, phi
};

struct Attitude {
    float R[9], sps, cps, sth, cth, sph, cph;
};

// contraction of a gradient in the rotation's entries with dR / d(psi, theta, phi)
__device__ __forceinline__ void angles_of(const Attitude &A, const float a[9], float &ps, float &th, float &ph)
{
    const float *R = A.R;
    ps = fmaf(a[3], R[0], -a[0] * R[3]) + fmaf(a[4], R[1], -a[1] * R[4]) + fmaf(a[5], R[2], -a[2] * R[5]);
    const float t0 = fmaf(A.cth, fmaf(a[1], A.sph, a[2] * A.cph), -a[0] * A.sth);
    const float t1 = fmaf(A.cth, fmaf(a[4], A.sph, a[5] * A.cph), -a[3] * A.sth);
    const float t2 = fmaf(A.sth, fmaf(a[7], A.sph, a[8] * A.cph), a[6] * A.cth);
    th = fmaf(A.cps, t0, fmaf(A.sps, t1, -t2));
    ph = fmaf(a[1], R[2], -a[2] * R[1]) + fmaf(a[4], R[5], -a[5] * R[4]) + fmaf(a[7], R[8], -a[8] * R[7]);
}

// One wheel at the step's start state: its forces as the forward pass forms
// them, and their gradients by reverse differentiation of F_z.
__device__ __forceinline__ void wheel_lin(const Veh &V, const Terrain &T, const Attitude &A, const Cell &cx,
                                          const Cell &cy, unsigned base, float z, float zl, float vx, float vy,
                                          float vz, float wx, float wy, float wz, float rx, float ry, float k,
                                          float b, float Fs, float di, WheelGrad &w)
{
    const float *R = A.R;
    const float ox = fmaf(rx, R[0], fmaf(ry, R[1], -V.hR * R[2]));
    const float oy = fmaf(rx, R[3], fmaf(ry, R[4], -V.hR * R[5]));
    const float oz = fmaf(rx, R[6], fmaf(ry, R[7], -V.hR * R[8]));
    const float vix = fmaf(-wz, ry, fmaf(-wy, V.hR, vx));
    const float viy = fmaf(wx, V.hR, fmaf(wz, rx, vy));
    const float viz = fmaf(-wy, rx, fmaf(wx, ry, vz));
    // the lookup; a query at or beyond the map's last node is clamped: what
    // moves it does not move the interpolation
    const float ux = fmaf(ox, T.inv_cell, cx.fc), uy = fmaf(oy, T.inv_cell, cy.fc);
    const bool inx = ux >= cx.lo && ux < cx.hi, iny = uy >= cy.lo && uy < cy.hi;
    bool off = false;
    float wa, wb;
    const float ix = axis(cx, ux, wa, off), iy = axis(cy, uy, wb, off);
    const unsigned o = texel_index(base, ix, iy, T.nx);
    const float4 *r0 = T.tex + o, *r1 = T.tex + (size_t)(o + (unsigned)T.nx);
    const float4 t00 = __ldg(r0), t10 = __ldg(r0 + 1), t01 = __ldg(r1), t11 = __ldg(r1 + 1);
    const float4 t = lerp4(t00, t10, t01, t11, wa, wb, T.has_cm != 0);
    const float tx = fmaf(-R[3], t.z, fmaf(-R[0], t.y, R[6]));
    const float ty = fmaf(-R[4], t.z, fmaf(-R[1], t.y, R[7]));
    const float tz = fmaf(-R[5], t.z, fmaf(-R[2], t.y, R[8]));
    const float itz = rcp(tz);
    const float Q = (z - t.x) + (oz + zl);
    const float chi = Q * itz;
    const float a = fmaf(-chi, wy, vix), bv = fmaf(chi, wx, viy);
    const float num = fmaf(tz, viz, fmaf(ty, bv, tx * a));
    const float chid = num * itz;
    const float Fk = fmaxf(fmaf(-k, chi, Fs), 0.f);
    const float Fb = fmaf(-b, chid, Fk);
    w.Fz = Fk > 0.f ? fmaxf(Fb, 0.f) : 0.f;
    const float Ca = V.C * (atan2_r(viy, vix) - di);
    const float is = rsq(fmaf(Ca, Ca, V.mu2));
    w.ratio = (-Ca * V.mu) * is;
    w.Fy = w.Fz * w.ratio;
    // slip: F_z dT / dCa dCa / dalpha, T' = -mu^3 / (mu^2 + Ca^2)^(3/2),
    // alpha = atan2(viy, vix) - di
    const float dT = w.Fz * (-V.mu * V.mu2 * is * is * is * V.C);
    const float r2 = fmaf(vix, vix, viy * viy);
    const float ir2 = r2 > 0.f ? rcp(r2) : 0.f;
    const float ax = -dT * viy * ir2, ay = dT * vix * ir2;      // by vix, viy
    w.a[0] = ax;
    w.a[1] = ay;
    w.a[2] = ay * V.hR;
    w.a[3] = -ax * V.hR;
    w.a[4] = fmaf(ay, rx, -ax * ry);
    w.ad = -dT;
    // suspension: F_z = F_k - b chid while both are positive, F_k = F_s - k chi
    const bool on = Fk > 0.f && Fb > 0.f;
    const float aN = on ? -b * itz : 0.f;                        // by num
    float aItz = on ? -b * num : 0.f;
    const float aA = aN * tx, aB = aN * ty, aViz = aN * tz;
    const float aChi = (on ? -k : 0.f) - aA * wy + aB * wx;
    const float aQ = aChi * itz;
    aItz = fmaf(aChi, Q, aItz);
    const float aTx = aN * a, aTy = aN * bv, aTz = fmaf(-aItz * itz, itz, aN * viz);
    // tau = R^T (-f_x, -f_y, 1), the height and the slopes through the lookup
    const float gx = -(aTx * R[0] + aTy * R[1] + aTz * R[2]);
    const float gy = -(aTx * R[3] + aTy * R[4] + aTz * R[5]);
    const float oa = 1.f - wa, ob = 1.f - wb;
    const float da_f = ob * (t10.x - t00.x) + wb * (t11.x - t01.x), db_f = oa * (t01.x - t00.x) + wa * (t11.x - t10.x);
    const float da_x = ob * (t10.y - t00.y) + wb * (t11.y - t01.y), db_x = oa * (t01.y - t00.y) + wa * (t11.y - t10.y);
    const float da_y = ob * (t10.z - t00.z) + wb * (t11.z - t01.z), db_y = oa * (t01.z - t00.z) + wa * (t11.z - t10.z);
    const float aOx = inx ? (-aQ * da_f + gx * da_x + gy * da_y) * T.inv_cell : 0.f;
    const float aOy = iny ? (-aQ * db_f + gx * db_x + gy * db_y) * T.inv_cell : 0.f;
    const float aR[9] = {fmaf(aOx, rx, -aTx * t.y), fmaf(aOx, ry, -aTy * t.y), fmaf(-aOx, V.hR, -aTz * t.y),
                         fmaf(aOy, rx, -aTx * t.z), fmaf(aOy, ry, -aTy * t.z), fmaf(-aOy, V.hR, -aTz * t.z),
                         fmaf(aQ, rx, aTx), fmaf(aQ, ry, aTy), fmaf(-aQ, V.hR, aTz)};
    w.g[0] = aOx;
    w.g[1] = aOy;
    w.g[2] = aQ;
    angles_of(A, aR, w.g[3], w.g[4], w.g[5]);
    w.g[6] = aA;
    w.g[7] = aB;
    w.g[8] = aViz;
    w.g[9] = fmaf(aB, V.hR, fmaf(aViz, ry, aB * chi));
    w.g[10] = -fmaf(aA, V.hR, fmaf(aViz, rx, aA * chi));
    w.g[11] = fmaf(aB, rx, -aA * ry);
    // costmap rate
    w.c[0] = w.c[1] = w.c[2] = w.c[3] = w.c[4] = w.c[5] = 0.f;
    if (T.has_cm) {
        const float da_c = ob * (t10.w - t00.w) + wb * (t11.w - t01.w), db_c = oa * (t01.w - t00.w) + wa * (t11.w - t10.w);
        const float px = inx ? da_c * T.inv_cell : 0.f, py = iny ? db_c * T.inv_cell : 0.f;
        const float cR[9] = {px * rx, px * ry, -px * V.hR, py * rx, py * ry, -py * V.hR, 0.f, 0.f, 0.f};
        w.c[0] = px;
        w.c[1] = py;
        angles_of(A, cR, w.c[3], w.c[4], w.c[5]);
    }
}

// dU_ESM / d(theta, phi): U = +/- M g Rbar (1 - (sin|phi| cos phibar + cos phi
// sin phibar)) cos theta
__device__ __forceinline__ void esm_grad(const Veh &V, float ph, float sth, float cth, float sph, float cph, float &th,
                                         float &dph)
{
    const float sg = fabsf(ph) < V.tip ? V.MgRbar : -V.MgRbar;
    const float sabs = ph < 0.f ? -sph : sph;
    const float sv = fmaf(sabs, V.cpb, cph * V.spb);
    th = -sg * (1.f - sv) * sth;
    dph = -sg * cth * ((ph < 0.f ? -V.cpb : V.cpb) * cph - V.spb * sph);
}

struct BackParams {
    Veh V;
    Cost C;
    Terrain T;
    const float2 *ctrl;       // [H][K]
    int K, n_sub;
    float h;
    int objective;
    int k0, k1;               // this segment's control steps
    int last, first;          // the rollout's last segment; its first
    const float4 *rec;        // [K][(k1 - k0) n_sub][4]
    const int *n_done, *emin;
    const float4 *fin;
    float *lam;               // [K][16] the adjoint between segments
    float *grad;              // [H][K][2]
};

// The columns of Euler step e of candidate j into `out`.
__device__ __forceinline__ void linearise(const BackParams &p, int j, int e, float *out)
{
    const Veh &V = p.V;
    const Cost &Cc = p.C;
    const Terrain &T = p.T;
    const float h = p.h;
    const int n_rec = (p.k1 - p.k0) * p.n_sub;
    const float4 *rec = p.rec + ((size_t)j * n_rec + (e - p.k0 * p.n_sub)) * 4;
    const float4 s0 = rec[0], s1 = rec[1], s2 = rec[2], s3 = rec[3];
    const float th = s1.w, ph = s2.x, d = s2.y, vx = s2.z, vy = s2.w, vz = s3.x, wx = s3.y, wy = s3.z, wz = s3.w;
    const float2 u = __ldg(p.ctrl + (size_t)(e / p.n_sub) * p.K + j);
    const bool inside = !(u.x < -V.ddmax || u.x > V.ddmax);       // as the clamp
    const float dd = clamp_keep_nan(u.x, -V.ddmax, V.ddmax);
    const float dn = fmaf(h, dd, d);
    const bool d_clamped = dn < -V.dmax || dn > V.dmax;
    Attitude A;
    float sd, cd;
    sincos_r(s1.z, A.sps, A.cps);
    sincos_r(th, A.sth, A.cth);
    sincos_r(ph, A.sph, A.cph);
    sincos_r(d, sd, cd);
    const float sth = A.sth, cth = A.cth, sph = A.sph, cph = A.cph;
    const float *R = A.R;
    rotation(A.sps, A.cps, sth, cth, sph, cph, A.R);
    const Cell cx = cell_of<false>(s0.x, s0.y, T.inv_cell, T.nx), cy = cell_of<false>(s0.z, s0.w, T.inv_cell, T.ny);
    const unsigned base = texel_base(cx, cy, T.nx);

    // gradients of the five force sums S = sum F_y (turned by delta in front),
    // sum F_z, sum r_y F_z, sum -r_x F_z, sum r_x F_y
    float S[5][12], Sd0 = 0.f, Sd4 = 0.f, cg[6];
#pragma unroll
    for (int c = 0; c < 12; ++c) S[0][c] = S[1][c] = S[2][c] = S[3][c] = S[4][c] = 0.f;
#pragma unroll
    for (int c = 0; c < 6; ++c) cg[c] = 0.f;
#pragma unroll 1
    for (int i = 0; i < 4; ++i) {
        const bool front = i < 2;
        const float rx = front ? V.Lf : -V.Lr, ry = (i & 1) ? -V.he : V.he;
        WheelGrad w;
        wheel_lin(V, T, A, cx, cy, base, s1.x, s1.y, vx, vy, vz, wx, wy, wz, rx, ry, front ? V.kf : V.kr,
                  front ? V.bf : V.br, front ? V.Fsf : V.Fsr, front ? d : 0.f, w);
        const float turn = front ? cd : 1.f;
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            float fy = w.ratio * w.g[c];
            if (c == 6) fy += w.a[0];
            if (c == 7) fy += w.a[1];
            if (c >= 9) fy += w.a[c - 7];
            fy *= turn;
            S[0][c] += fy;
            S[1][c] += w.g[c];
            S[2][c] = fmaf(ry, w.g[c], S[2][c]);
            S[3][c] = fmaf(-rx, w.g[c], S[3][c]);
            S[4][c] = fmaf(rx, fy, S[4][c]);
        }
        if (front) {
            const float fd = fmaf(w.ad, cd, -sd * w.Fy);
            Sd0 += fd;
            Sd4 = fmaf(rx, fd, Sd4);
        }
#pragma unroll
        for (int c = 0; c < 6; ++c) cg[c] += w.c[c];
    }
    // the force rows of the step's matrix (times the Euler step): y and z
    // velocity, then the rates by Euler's equations
    const float kv = h * V.invM, kx = h * V.invJxx, ky = h * V.invJyy, kz = h * V.invJzz;
    const float fx = -2.f * V.hR * ky * V.halfM;            // the rear constraint force in My
    float D[5][12];
#pragma unroll
    for (int c = 0; c < 12; ++c) {
        D[0][c] = kv * S[0][c];
        D[1][c] = kv * S[1][c];
        D[2][c] = kx * fmaf(V.hR, S[0][c], S[2][c]);
        D[3][c] = ky * S[3][c];
        D[4][c] = kz * S[4][c];
    }
    const float hg = h * V.g;
    D[0][4] = fmaf(hg, sth * sph, D[0][4]);                 // gravity in B
    D[0][5] = fmaf(-hg, cth * cph, D[0][5]);
    D[1][4] = fmaf(hg, cph * sth, D[1][4]);
    D[1][5] = fmaf(hg, sph * cth, D[1][5]);
    D[3][4] = fmaf(-fx * V.g, cth, D[3][4]);
    D[0][6] = fmaf(-h, wz, D[0][6]);                        // the velocities' cross terms
    D[0][8] = fmaf(h, wx, D[0][8]);
    D[0][9] = fmaf(h, vz, D[0][9]);
    D[0][11] = fmaf(-h, vx, D[0][11]);
    D[1][6] = fmaf(h, wy, D[1][6]);
    D[1][7] = fmaf(-h, wx, D[1][7]);
    D[1][9] = fmaf(-h, vy, D[1][9]);
    D[1][10] = fmaf(h, vx, D[1][10]);
    D[2][10] = fmaf(kx * V.dJyz, wz, D[2][10]);
    D[2][11] = fmaf(kx * V.dJyz, wy, D[2][11]);
    D[3][7] = fmaf(-fx, wz, D[3][7]);
    D[3][8] = fmaf(fx, wy, D[3][8]);
    D[3][9] = fmaf(-ky * V.dJxz, wz, D[3][9]);
    D[3][10] = fmaf(fx, vz, D[3][10]);
    D[3][11] = fmaf(-ky * V.dJxz, wx, fmaf(-fx, vy, D[3][11]));
    D[4][9] = fmaf(kz * V.dJxy, wy, D[4][9]);
    D[4][10] = fmaf(kz * V.dJxy, wx, D[4][10]);

    // the constants: the running cost's gradient, or the margin's at its state
    const float sv = fmaf(ph < 0.f ? -sph : sph, V.cpb, cph * V.spb);
    const float uu = V.MgRbar * (1.f - sv) * cth;
    const float U = fabsf(ph) < V.tip ? uu : -uu;
    const float soft = fmaxf(fmaf(-U, Cc.inv_eps, 1.f), 0.f);
    float eth, eph;
    esm_grad(V, ph, sth, cth, sph, cph, eth, eph);
    const bool cost = p.objective == kGradCost;
    const float aU = cost ? (soft > 0.f ? -h * 2.f * Cc.sigma * soft * Cc.inv_eps : 0.f)
                          : (e == p.emin[j] ? 1.f : 0.f);
    const float hc = cost ? h : 0.f;
    float cst[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) cst[c] = hc * cg[c];
    if (aU != 0.f) {
        cst[4] = fmaf(aU, eth, cst[4]);
        cst[5] = fmaf(aU, eph, cst[5]);
    }

    // the kinematic rows, and every column into shared memory
    const float ic = rcp(cth);
    const float wsc = fmaf(sph, wy, cph * wz), wdf = fmaf(cph, wy, -sph * wz);
    const float bth = fmaf(sph, vy, cph * vz);              // along dR / d(theta)
    const float xth = fmaf(cth, bth, -sth * vx), zth = -fmaf(sth, bth, cth * vx);
    float4 *o = (float4 *)out;
    const auto column = [&](int c, float x, float y, float z, float ps, float t, float f, float k) {
        o[4 * c] = make_float4(x, y, z, ps);
        o[4 * c + 1] = make_float4(t, f, 0.f, D[0][c]);
        o[4 * c + 2] = make_float4(D[1][c], D[2][c], D[3][c], D[4][c]);
        o[4 * c + 3] = make_float4(0.f, k, 0.f, 1.f);
    };
    column(X, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, cst[0]);
    column(Y, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, cst[1]);
    column(Z, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, cst[2]);
    column(PSI, -h * fmaf(R[5], vz, fmaf(R[4], vy, R[3] * vx)), h * fmaf(R[2], vz, fmaf(R[1], vy, R[0] * vx)), 0.f, 0.f,
           0.f, 0.f, cst[3]);
    column(TH, h * A.cps * xth, h * A.sps * xth, h * zth, h * wsc * sth * ic * ic, 0.f,
           h * wsc * fmaf(sth * ic, sth * ic, cth * ic), cst[4]);
    column(PH, h * fmaf(R[2], vy, -R[1] * vz), h * fmaf(R[5], vy, -R[4] * vz), h * fmaf(R[8], vy, -R[7] * vz),
           h * ic * wdf, -h * wsc, h * sth * ic * wdf, cst[5]);
    column(VX, h * R[0], h * R[3], h * R[6], 0.f, 0.f, 0.f, 0.f);
    column(VY, h * R[1], h * R[4], h * R[7], 0.f, 0.f, 0.f, 0.f);
    column(VZ, h * R[2], h * R[5], h * R[8], 0.f, 0.f, 0.f, 0.f);
    column(WX, 0.f, 0.f, 0.f, 0.f, 0.f, h, 0.f);
    column(WY, 0.f, 0.f, 0.f, h * sph * ic, h * cph, h * sph * sth * ic, 0.f);
    column(WZ, 0.f, 0.f, 0.f, h * cph * ic, -h * sph, h * cph * sth * ic, 0.f);
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    o[4 * DE] = zero;
    o[4 * DE + 1] = make_float4(0.f, 0.f, 0.f, kv * Sd0);
    o[4 * DE + 2] = make_float4(0.f, kx * V.hR * Sd0, 0.f, kz * Sd4);
    o[4 * DE + 3] = make_float4(0.f, 0.f, 0.f, d_clamped ? 0.f : 1.f);
    o[4 * kGdd] = zero;
    o[4 * kGdd + 1] = zero;
    o[4 * kGdd + 2] = zero;
    o[4 * kGdd + 3] = make_float4(d_clamped ? 0.f : h, hc * 2.f * Cc.wc * dd, inside ? 1.f : 0.f, 1.f);
    o[4 * kGax] = zero;
    o[4 * kGax + 1] = make_float4(0.f, 0.f, h, 0.f);
    o[4 * kGax + 2] = make_float4(0.f, 0.f, fx, 0.f);
    o[4 * kGax + 3] = make_float4(0.f, 0.f, 0.f, 1.f);
}

// The recursion over n steps from the last to step e of `mats`, this lane's
// column of each: returns the adjoint (and the open gradients) before them.
// SPAN lanes run one candidate; candidates with fewer steps than the warp's
// longest sit out the rest.  The adjoint goes round through 16 floats of
// shared memory, in turn the two of `turn`: one store and four broadcast loads
// a step, where 13 shuffles took twice the time.  GUARD leaves out the
// matrix's zeros, which a NaN would pass through.
template <int SPAN, bool GUARD>
__device__ __forceinline__ float recursion(const BackParams &p, int j, const float *mats, float *turn, int e, int n,
                                           int lane, float lam)
{
    const int col = lane < kCols ? lane : kCols - 1;
    const int n_max = SPAN == 32 ? n : max(n, __shfl_xor_sync(kFull, n, 16));
    int k = (e + n - 1) / p.n_sub, sub = (e + n - 1) - k * p.n_sub;
    const float4 *m = (const float4 *)mats + (size_t)max(n - 1, 0) * (kStepFloats / 4) + 4 * col;
    float4 a = m[0], b = m[1], c = m[2], d = m[3];
    for (int s = 0; s < n_max; ++s) {
        float *l = turn + (s & 1) * 16;
        if (SPAN == 16 || lane < 16) l[lane] = lam;
        const float4 a0 = a, b0 = b, c0 = c, d0 = d;
        if (s + 1 < n) {                                    // the next step's column, ahead
            m -= kStepFloats / 4;
            a = m[0]; b = m[1]; c = m[2]; d = m[3];
        }
        __syncwarp();
        const float4 la = ((const float4 *)l)[0], lb = ((const float4 *)l)[1], lc = ((const float4 *)l)[2];
        const float ld = l[DE];
        const auto add = [](float w, float v, float q) { return GUARD && w == 0.f ? q : fmaf(w, v, q); };
        float q0 = add(a0.x, la.x, d0.y), q1 = add(a0.y, la.y, 0.f), q2 = add(a0.z, la.z, 0.f), q3 = add(a0.w, la.w, 0.f);
        q0 = add(b0.x, lb.x, q0);
        q1 = add(b0.y, lb.y, q1);
        q2 = add(b0.z, lb.z, q2);
        q3 = add(b0.w, lb.w, q3);
        q0 = add(c0.x, lc.x, q0);
        q1 = add(c0.y, lc.y, q1);
        q2 = add(c0.z, lc.z, q2);
        q3 = add(c0.w, lc.w, q3);
        q0 = add(d0.x, ld, q0);
        const float q = (q0 + q1) + (q2 + q3);
        if (SPAN == 32 || s < n) {
            lam = GUARD && d0.w == 0.f ? q : fmaf(d0.w, lam, q);
            if (sub-- == 0) {                               // the control step is complete
                if (lane == kGdd || lane == kGax)
                    p.grad[((size_t)k * p.K + j) * 2 + (lane - kGdd)] = lane == kGdd && d0.z == 0.f ? 0.f : lam;
                if (lane >= kGdd) lam = 0.f;
                --k;
                sub = p.n_sub - 1;
            }
        }
    }
    __syncwarp();
    return lam;
}

// a chunk's recursion; a diverged rollout's infinities and NaN pass only
// through the entries the steps' matrices have
template <int SPAN>
__device__ __forceinline__ float run_chunk(const BackParams &p, int j, const float *mats, float *turn, int e, int n,
                                           int lane, float lam)
{
    const float out = recursion<SPAN, false>(p, j, mats, turn, e, n, lane, lam);
    return __any_sync(kFull, !isfinite(out)) ? recursion<SPAN, true>(p, j, mats, turn, e, n, lane, lam) : out;
}

// What the recursion of candidate j starts from; lane is the component.
__device__ __forceinline__ float first_lam(const BackParams &p, int j, int n_done, int lane)
{
    float lam = 0.f;
    if (!p.last) return lane < kRows ? p.lam[(size_t)j * 16 + lane] : 0.f;
    const float4 f = p.fin[j];
    if (p.objective == kGradCost) {
        // terminal cost w_g |p_xy - goal|
        const float dist = sqrtf(fmaf(f.x, f.x, f.y * f.y));
        if (dist > 0.f && lane < 2) lam = p.C.wg * (lane == 0 ? f.x : f.y) / dist;
    } else if (p.emin[j] == n_done) {
        // the final state holds the margin
        float sth, cth, sph, cph, t, f5;
        sincos_r(f.z, sth, cth);
        sincos_r(f.w, sph, cph);
        esm_grad(p.V, f.w, sth, cth, sph, cph, t, f5);
        if (lane == TH) lam = t;
        if (lane == PH) lam = f5;
    }
    return lam;
}

// gradients of the segment's control steps that never ran
__device__ __forceinline__ void zero_grad(const BackParams &p, int j, int n_done, int t, int nt)
{
    for (int k = max(p.k0, (n_done + p.n_sub - 1) / p.n_sub) + t; k < p.k1; k += nt)
        *(float2 *)(p.grad + ((size_t)k * p.K + j) * 2) = make_float2(0.f, 0.f);
}

// A few candidates: one per CTA.  kWide warps linearise a chunk of 32 kWide
// steps into one of two buffers (976 bytes a step: the SM's shared memory)
// while another warp runs the recursion over the chunk after it.
constexpr int kWide = 3;
__global__ void __launch_bounds__(32 * (kWide + 1)) grad_back_wide_kernel(const __grid_constant__ BackParams p)
{
    extern __shared__ __align__(16) float mats[];           // [2][32 kWide][kStepFloats], [2][16]
    constexpr int kChunk = 32 * kWide;
    const int j = blockIdx.x, t = threadIdx.x, lane = t & 31;
    const bool runs = t >= kChunk;
    const int n_done = p.n_done[j];
    const int e0 = p.k0 * p.n_sub, e1 = min(p.k1 * p.n_sub, n_done);
    zero_grad(p, j, n_done, t, 32 * (kWide + 1));
    float lam = runs ? first_lam(p, j, n_done, lane) : 0.f;
    const int n = e1 > e0 ? (e1 - e0 + kChunk - 1) / kChunk : 0;
    for (int i = 0; i <= n; ++i) {
        if (!runs && i < n) {
            const int hi = e1 - i * kChunk, e = max(e0, hi - kChunk) + t;
            if (e < hi) linearise(p, j, e, mats + (size_t)((i & 1) * kChunk + t) * kStepFloats);
        }
        if (runs && i > 0) {
            const int hi = e1 - (i - 1) * kChunk, lo = max(e0, hi - kChunk);
            lam = run_chunk<32>(p, j, mats + (size_t)((i - 1) & 1) * kChunk * kStepFloats,
                                mats + (size_t)2 * kChunk * kStepFloats, lo, hi - lo, lane, lam);
        }
        __syncthreads();
    }
    if (runs && !p.first && lane < kRows) p.lam[(size_t)j * 16 + lane] = lam;
}

// Many candidates: two per warp.  The warp linearises 16 steps of each, then
// its halves run the two recursions side by side.  Seven warps fit the SM's
// shared memory; the warps cover one another's phases.
__global__ void __launch_bounds__(32) grad_back_kernel(const __grid_constant__ BackParams p)
{
    extern __shared__ __align__(16) float mats[];           // [2][16][kStepFloats], [2][2][16]
    const int half = threadIdx.x >> 4, lane = threadIdx.x & 15;
    const int j = min(2 * (int)blockIdx.x + half, p.K - 1);
    const bool live = 2 * (int)blockIdx.x + half < p.K;
    const int n_done = p.n_done[j];
    const int e0 = p.k0 * p.n_sub, e1 = live ? min(p.k1 * p.n_sub, n_done) : 0;
    if (live) zero_grad(p, j, n_done, lane, 16);
    float lam = first_lam(p, j, n_done, lane);
    float *mine = mats + (size_t)half * 16 * kStepFloats;
    for (int hi = e1; __any_sync(kFull, hi > e0); hi -= 16) {
        const int lo = max(e0, hi - 16);
        if (lo + lane < hi) linearise(p, j, lo + lane, mine + (size_t)lane * kStepFloats);
        __syncwarp();
        lam = run_chunk<16>(p, j, mine, mats + 32 * kStepFloats + half * 32, lo, max(hi - lo, 0), lane, lam);
        __syncwarp();
    }
    if (live && !p.first && lane < kRows) p.lam[(size_t)j * 16 + lane] = lam;
}

template <int LANES, bool PER_X0>
__global__ void __launch_bounds__(kPlanBlock, LANES == 4 ? 1 : LANES == 2 ? 8 : 6)
grad_forward_kernel(const __grid_constant__ PlanParams p, const __grid_constant__ Trace tr)
{
    __shared__ Duo<LANES> sh;
    int j;
    float J = 0.f, margin = CUDART_INF_F;
    bool feasible = false;
    duo_rollout<LANES, PER_X0, TEX_F32, kAccF32>(p, tr, sh, blockIdx.x, j, J, margin, feasible);
}

template <bool PER_X0>
void launch_forward(const PlanParams &p, const Trace &tr, cudaStream_t stream)
{
    int layout = plan_layout(0, p.N);
    if (layout == kLayoutOne) layout = kLayoutDuo1;         // the trace is a two-warp rollout's
    const unsigned grid = (unsigned)layout_ctas(layout, p.N);
    if (layout == kLayoutDuo4) grad_forward_kernel<4, PER_X0><<<grid, kPlanBlock, 0, stream>>>(p, tr);
    else if (layout == kLayoutDuo2) grad_forward_kernel<2, PER_X0><<<grid, kPlanBlock, 0, stream>>>(p, tr);
    else grad_forward_kernel<1, PER_X0><<<grid, kPlanBlock, 0, stream>>>(p, tr);
}

// candidates up to which a CTA takes one: two waves of one CTA per SM, where the
// two forms meet (202 us for 300 candidates of 330 steps, one per CTA; 190 us
// for 305 of 240, two per warp)
constexpr int kBackWideMaxK = 304;

cudaError_t launch_back(const BackParams &b, cudaStream_t stream)
{
    if (b.K <= kBackWideMaxK) {
        constexpr int kSmem = (2 * 32 * kWide * kStepFloats + 32) * (int)sizeof(float);
        const cudaError_t e = cudaFuncSetAttribute(grad_back_wide_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   kSmem);
        if (e != cudaSuccess) return e;
        grad_back_wide_kernel<<<(unsigned)b.K, 32 * (kWide + 1), kSmem, stream>>>(b);
    } else {
        grad_back_kernel<<<(unsigned)((b.K + 1) / 2), 32, (32 * kStepFloats + 64) * sizeof(float), stream>>>(b);
    }
    return cudaGetLastError();
}

// Bytes of one candidate: a record of the trace, a checkpoint, the adjoint
// between segments, and what the forward pass leaves of its end.
constexpr size_t kRecBytes = 64, kCkptBytes = 20 * sizeof(float), kLamBytes = 16 * sizeof(float),
                 kEndBytes = sizeof(float4) + 2 * sizeof(int);
// What `ckpt` bounds the workspace by, in bytes per candidate: a state in each
// of four lanes, times the control steps' checkpoints and two segments' Euler
// steps (one where two would take more than kTwoBytes).
constexpr size_t kStateBytes = 4 * 20 * sizeof(float);

}  // namespace

GradPlan grad_plan(int K, int H, int n_sub, int ckpt)
{
    const auto up = [](size_t v) { return (v + 255) / 256 * 256; };
    const size_t per_step = (size_t)n_sub * kRecBytes;      // of one candidate's trace, per control step
    const auto segments = [&](size_t seg) { return (H + seg - 1) / seg; };
    const auto bytes = [&](size_t seg) {
        const size_t n = segments(seg);
        return seg * per_step + kEndBytes + (n > 1 ? n * kCkptBytes + kLamBytes : 0);
    };
    // what `ckpt` allows, and the most control steps that fit it: ckpt do
    const auto allowed = [&](int b) { return kStateBytes * (segments(ckpt) + (size_t)b * ckpt * n_sub); };
    const size_t bound = std::max(allowed(1), std::min(allowed(2), kTwoBytes / K));
    size_t seg = std::min(std::max(bound / per_step, (size_t)ckpt), (size_t)H);
    while (seg > (size_t)ckpt && bytes(seg) > bound) --seg;
    if (H * per_step <= kWholeBytes / K) seg = H;
    GradPlan g;
    g.n_seg = (int)segments(seg);
    g.seg = (int)segments(g.n_seg);                         // of one length, but for the last
    g.n_seg = (int)segments(g.seg);
    size_t o = 0;
    g.rec = o;  o = up(o + per_step * g.seg * K);
    g.ckpt = o; o = up(o + (g.n_seg > 1 ? (size_t)g.n_seg * K * kCkptBytes : 0));
    g.fin = o;  o = up(o + (size_t)K * sizeof(float4));
    g.lam = o;  o = up(o + (g.n_seg > 1 ? (size_t)K * kLamBytes : 0));
    g.ints = o; o = up(o + (size_t)K * 2 * sizeof(int));
    g.total = o;
    return g;
}

cudaError_t launch_grad(const PlanParams &p, const GradPlan &g, int objective, char *buf, float *grad,
                        cudaStream_t stream)
{
    Trace tr;
    tr.rec = (float4 *)(buf + g.rec);
    tr.seg = g.seg;
    tr.objective = objective;
    tr.fin = (float4 *)(buf + g.fin);
    tr.n_done = (int *)(buf + g.ints);
    tr.emin = tr.n_done + p.N;
    BackParams b;
    b.V = p.V;
    b.C = p.C;
    b.T = p.T;
    b.ctrl = p.ctrl;
    b.K = p.N;
    b.n_sub = p.n_sub;
    b.h = p.h;
    b.objective = objective;
    b.rec = tr.rec;
    b.n_done = tr.n_done;
    b.emin = tr.emin;
    b.fin = tr.fin;
    b.lam = (float *)(buf + g.lam);
    b.grad = grad;
    for (int s = g.n_seg - 1; s >= 0; --s) {
        const bool last = s == g.n_seg - 1;
        // the whole rollout with the last segment's trace and the checkpoints,
        // then each earlier segment from its checkpoint
        tr.k0 = last ? 0 : s * g.seg;
        tr.k1 = last ? p.H : (s + 1) * g.seg;
        tr.trace_k0 = s * g.seg;
        float *ckpt = (float *)(buf + g.ckpt);
        tr.ckpt = last && g.n_seg > 1 ? ckpt : nullptr;
        tr.from = last ? nullptr : ckpt + (size_t)s * 20 * p.N;
        if (p.x0_soa) launch_forward<true>(p, tr, stream);
        else launch_forward<false>(p, tr, stream);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        b.k0 = s * g.seg;
        b.k1 = tr.k1;
        b.last = last;
        b.first = s == 0;
        e = launch_back(b, stream);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace atp
