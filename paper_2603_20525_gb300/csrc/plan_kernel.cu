// plan_kernel.cu - fused SRB rollout, cost, ESM margin and empirical argmin
// (arxiv 2603.20525, Sec. IV-A..IV-D) for sm_103a.
//
// Design
//   * A full GPU runs one thread per candidate (rollout_one).  Below that the
//     time is one candidate's chain of dependent instructions, and two warps
//     share a group of candidates (the two-warp layouts below), with one, two
//     or four lanes of each warp per candidate by batch size.  The state
//     stays in registers for the whole horizon; per Euler step the only
//     global memory traffic is 16 terrain texels (four bilinear lookups of
//     one float4 per corner) through the read-only path, which the L1 and the
//     129 MB L2 serve for every terrain size used.
//   * Every layout forms every quantity by the same expressions in the same
//     order, so all of them give the same bits.
//   * Controls are time-major float2 [H][N]: a warp reads one coalesced 256 B
//     line per control step.
//   * The reduction is fused into the tail: a warp-shuffle min of a packed
//     64-bit key (infeasible bit, order-preserving image of the FP32 cost,
//     candidate index), one shared-memory step per CTA, one 64-bit atomicMin
//     per CTA, a ballot/popc feasible count, and a ticket that elects the last
//     CTA to write the result and the best candidate's controls (and, when
//     asked for, its per-step margins).
#include "duo.cuh"
#include "plan_kernel.cuh"
#include "plan_tail.cuh"

#include <cuda_bf16.h>
#include <math_constants.h>

namespace atp {

// One thread per candidate.  The four sincos take the reduction without a
// branch, one test covering their slow form: headings spread over the circle
// and tipped candidates' roll and pitch grow, so that warps ran both paths of
// each (paper configuration 4.84 -> 4.41 ms, 50000 x 100 x 4 steps 664 -> 639 us).
template <bool PER_X0, int TEX, int ACC>
__device__ __forceinline__ void rollout_one(const PlanParams &p, int j, float &J, float &margin, bool &feasible)
{
    const Veh &V = p.V;
    const Cost &Cc = p.C;
    const Terrain &T = p.T;
    {
        // state; x, y relative to the terrain origin; *_l are the low parts of
        // the compensated components
        float x, xl, y, yl, z, zl, psi, psil, vx, vxl, vy, vyl, vz, vzl;
        float th, ph, wx, wy, wz, d;
        {
            float x0[13];
            if (PER_X0) {
                const size_t N = (size_t)p.N;
#pragma unroll
                for (int c = 0; c < 13; ++c) x0[c] = p.x0_soa[c * N + j];
            } else {
#pragma unroll
                for (int c = 0; c < 13; ++c) x0[c] = p.x0[c];
            }
            two_sum(x0[0], -T.x0_hi, x, xl);
            xl -= T.x0_lo;
            two_sum(x0[1], -T.y0_hi, y, yl);
            yl -= T.y0_lo;
            z = x0[2]; psi = x0[3]; th = x0[4]; ph = x0[5];
            vx = x0[6]; vy = x0[7]; vz = x0[8];
            wx = x0[9]; wy = x0[10]; wz = x0[11]; d = x0[12];
            zl = psil = vxl = vyl = vzl = 0.f;
        }
        bool done = false, off = false;
        const float h = p.h;
        const bool acc64 = ACC == kAccRuntime ? p.acc64 != 0 : ACC == kAccF64;
        double J64 = 0.0;          // the running cost in FP64 when acc64
        float Ufrozen = 0.f;
        // the smallest per-step margin so far, its control step (first on
        // ties), and the last step's margin, which the final state joins
        float msm = CUDART_INF_F, last_sm = CUDART_INF_F;
        int mstep = 0;

        for (int k = 0; k < p.H; ++k) {
            // zero-order hold; admissible steering rate |delta_dot| <= max
            const float2 u = __ldg(p.ctrl + (size_t)k * p.N + j);
            // ask L1 for the next interval's control, which costs no register
            // (holding it in one costs more here than the latency saved)
            if (k + 1 < p.H)
                asm volatile("prefetch.global.L1 [%0];" ::"l"(p.ctrl + (size_t)(k + 1) * p.N + j));
            const float dd = clamp_keep_nan(u.x, -V.ddmax, V.ddmax);
            const float ax = u.y;
            float sm = CUDART_INF_F;
            for (int sub = 0; sub < p.n_sub; ++sub) {
                if (done) {            // frozen at the goal: the same state each step
                    sm = fminf(sm, Ufrozen);
                    continue;
                }
                float sps, cps, sth, cth, sph, cph;
                float sd, cd;
                sincos_g<false>(d, sd, cd);
                sincos_g<false>(psi, sps, cps);
                sincos_g<false>(th, sth, cth);
                sincos_g<false>(ph, sph, cph);
                if (fmaxf(fmaxf(fabsf(psi), fabsf(d)), fmaxf(fabsf(th), fabsf(ph))) >= kSincosMax) {
                    sincos_g<true>(psi, sps, cps);
                    sincos_g<true>(th, sth, cth);
                    sincos_g<true>(ph, sph, cph);
                    sincos_g<true>(d, sd, cd);
                }
                const float U = esm(V, ph, sph, cph, cth);
                margin = fminf(margin, U);
                sm = fminf(sm, U);
                // goal test before the step (Sec. IV-C, reading Q4)
                const float gdx = (x - Cc.gx_hi) + (xl - Cc.gx_lo);
                const float gdy = (y - Cc.gy_hi) + (yl - Cc.gy_lo);
                if (fmaf(gdx, gdx, gdy * gdy) <= Cc.goal_r2) {
                    done = true;
                    Ufrozen = U;
                    continue;
                }
                // 3-2-1 rotation, body -> world (Sec. IV-A)
                Body B;
                float *R = B.R;
                rotation(sps, cps, sth, cth, sph, cph, R);
                B.cx = cell_of(x, xl, T.inv_cell, T.nx);
                B.cy = cell_of(y, yl, T.inv_cell, T.ny);
                B.base = texel_base(B.cx, B.cy, T.nx);
                off = off || off_com(B.cx, B.cy);
                B.z_hi = z;
                B.z_lo = zl;
                B.vx = vx; B.vy = vy; B.vz = vz;
                B.wx = wx; B.wy = wy; B.wz = wz;
                // gravity in B: R^T (0, 0, -g)
                const float gBx = -V.g * R[6], gBy = -V.g * R[7], gBz = -V.g * R[8];
                // summed forces and moments (Sec. IV-A); the rear
                // longitudinal constraint force enters My only
                const WheelOut fl = wheel<TEX>(V, T, B, V.Lf, V.he, V.kf, V.bf, V.Fsf, d, off);
                const WheelOut fr = wheel<TEX>(V, T, B, V.Lf, -V.he, V.kf, V.bf, V.Fsf, d, off);
                const WheelOut rl = wheel<TEX>(V, T, B, -V.Lr, V.he, V.kr, V.br, V.Fsr, 0.f, off);
                const WheelOut rr = wheel<TEX>(V, T, B, -V.Lr, -V.he, V.kr, V.br, V.Fsr, 0.f, off);
                const float Fyf = (fl.Fy + fr.Fy) * cd;
                const float Fyr = rl.Fy + rr.Fy;
                const float FyB = Fyf + Fyr;
                const float FzB = (fl.Fz + fr.Fz) + (rl.Fz + rr.Fz);
                const float Mx = fmaf(V.hR, FyB, V.he * ((fl.Fz - fr.Fz) + (rl.Fz - rr.Fz)));
                float My = -V.Lf * (fl.Fz + fr.Fz) + V.Lr * (rl.Fz + rr.Fz);
                const float Mz = V.Lf * Fyf + -V.Lr * Fyr;
                const float csum = (fl.cost + fr.cost) + (rl.cost + rr.cost);
                const float Fx = V.halfM * fmaf(-wz, vy, fmaf(wy, vz, ax - gBx));
                My = fmaf(-V.hR, 2.f * Fx, My);
                // running cost L = L_0 + L_soft (Sec. IV-C), left Riemann sum
                const float soft = fmaxf(fmaf(-U, Cc.inv_eps, 1.f), 0.f);
                const float L = fmaf(Cc.sigma * soft, soft, fmaf(Cc.wc * dd, dd, Cc.wt)) + csum;
                if (acc64) J64 += (double)(h * L);
                else J = fmaf(h, L, J);
                // state derivative A(xi) + B zeta (Sec. IV-A)
                const float ic = rcp(cth);
                const float wsc = fmaf(sph, wy, cph * wz);
                const float dx = fmaf(R[2], vz, fmaf(R[1], vy, R[0] * vx));
                const float dy = fmaf(R[5], vz, fmaf(R[4], vy, R[3] * vx));
                const float dz = fmaf(R[8], vz, fmaf(R[7], vy, R[6] * vx));
                const float dpsi = wsc * ic;
                const float dth = fmaf(cph, wy, -sph * wz);
                const float dph = fmaf(wsc, sth * ic, wx);
                const float dvy = fmaf(-wz, vx, fmaf(wx, vz, fmaf(FyB, V.invM, gBy)));
                const float dvz = fmaf(wy, vx, fmaf(-wx, vy, fmaf(FzB, V.invM, gBz)));
                const float dwx = fmaf(V.dJyz * wy, wz, Mx) * V.invJxx;
                const float dwy = fmaf(-V.dJxz * wx, wz, My) * V.invJyy;
                const float dwz = fmaf(V.dJxy * wx, wy, Mz) * V.invJzz;
                // forward Euler (Sec. IV-D), steering angle clamped (reading Q5)
                acc2(x, xl, h * dx);
                acc2(y, yl, h * dy);
                acc2(z, zl, h * dz);
                acc2(psi, psil, h * dpsi);
                acc2(vx, vxl, h * ax);
                acc2(vy, vyl, h * dvy);
                acc2(vz, vzl, h * dvz);
                th = fmaf(h, dth, th);
                ph = fmaf(h, dph, ph);
                wx = fmaf(h, dwx, wx);
                wy = fmaf(h, dwy, wy);
                wz = fmaf(h, dwz, wz);
                d = clamp_keep_nan(fmaf(h, dd, d), -V.dmax, V.dmax);
            }
            if (p.step_margin && k + 1 < p.H) p.step_margin[(size_t)k * p.N + j] = sm;
            if (k + 1 < p.H) {
                if (sm < msm) {
                    msm = sm;
                    mstep = k;
                }
            } else {
                last_sm = sm;
            }
        }
        // final state: margin, goal test, terminal cost Phi (Sec. IV-C)
        {
            float sth, cth, sph, cph;
            sincos_r(th, sth, cth);
            sincos_r(ph, sph, cph);
            const float U = esm(V, ph, sph, cph, cth);
            margin = fminf(margin, U);
            last_sm = fminf(last_sm, U);
            if (last_sm < msm) mstep = p.H - 1;
            if (p.step_margin) p.step_margin[(size_t)(p.H - 1) * p.N + j] = last_sm;
            const float gdx = (x - Cc.gx_hi) + (xl - Cc.gx_lo);
            const float gdy = (y - Cc.gy_hi) + (yl - Cc.gy_lo);
            const float d2 = fmaf(gdx, gdx, gdy * gdy);
            if (!done && d2 <= Cc.goal_r2) done = true;
            if (acc64) J = (float)(J64 + (double)(Cc.wg * sqrtf(d2)));
            else J = fmaf(Cc.wg, sqrtf(d2), J);
        }
        // fold the low parts back and leave the terrain frame
        const float xs[13] = {(x + T.x0_hi) + (xl + T.x0_lo), (y + T.y0_hi) + (yl + T.y0_lo),
                              z + zl, psi + psil, th, ph, vx + vxl, vy + vyl, vz + vzl,
                              wx, wy, wz, d};
        bool finite = isfinite(J);
#pragma unroll
        for (int c = 0; c < 13; ++c) finite = finite && isfinite(xs[c]);
        if (!finite) J = CUDART_INF_F;
        feasible = finite && margin > 0.f;
        const uint8_t fl = (feasible ? ATP_FLAG_FEASIBLE : 0) | (done ? ATP_FLAG_DONE : 0) |
                           (off ? ATP_FLAG_OFFMAP : 0) | (finite ? 0 : ATP_FLAG_NONFINITE);
        if (p.cost) p.cost[j] = J;
        if (p.margin) p.margin[j] = margin;
        if (p.flags) p.flags[j] = fl;
        if (p.min_step) p.min_step[j] = mstep;
        if (p.xf) {
            const size_t N = (size_t)p.N;
#pragma unroll
            for (int c = 0; c < 13; ++c) p.xf[c * N + j] = xs[c];
        }
    }

}

// Five CTAs per SM leave ptxas 168 registers and no spills: 2 % faster on the
// paper configuration than at six or seven (128 registers, 32 B of spills; the
// lookups' map edges keep more values live than the integer clamps they
// replaced) and 10 % than at four.
template <bool PER_X0, bool REDUCE, int TEX, int ACC>
__global__ void __launch_bounds__(kPlanBlock, 5)
plan_kernel(const __grid_constant__ PlanParams p)
{
    const int j = blockIdx.x * kPlanBlock + threadIdx.x;     // N <= 2^31 - 1025
    const bool live = j < p.N;
    float J = 0.f, margin = CUDART_INF_F;
    bool feasible = false;
    if (live) rollout_one<PER_X0, TEX, ACC>(p, j, J, margin, feasible);
    if (!REDUCE) return;
    plan_tail(p, j, live, J, feasible, gridDim.x);
}

// ---- the two-warp layouts (duo.cuh) -------------------------------------------

// Registers: one lane runs best free of spills (168 registers, six CTAs per
// SM: 0.296 ms at 16384 candidates against 0.345 ms at the 128-register cap),
// two and four lanes fit 128.
template <int LANES, bool PER_X0, bool REDUCE, int TEX, int ACC>
__global__ void __launch_bounds__(kPlanBlock, LANES == 4 ? 1 : LANES == 2 ? 8 : 6)
plan_duo_kernel(const __grid_constant__ PlanParams p)
{
    __shared__ Duo<LANES> sh;
    int j;
    float J = 0.f, margin = CUDART_INF_F;
    bool feasible = false;
    const bool leader = duo_rollout<LANES, PER_X0, TEX, ACC>(p, NoTrace{}, sh, blockIdx.x, j, J, margin, feasible);
    if (!REDUCE) return;
    plan_tail(p, j, leader, J, feasible, gridDim.x);
}

// Terrain staging: the one-lane rollout with a window of the texels in
// shared memory.  Every CTA copies the window (plain coalesced loads, once per
// CTA; at most 225 KB, so one CTA of 16 warps per SM), then each candidate
// reads the lookups inside it from shared memory and the rest through L1 as
// usual.  The texel values are the same either way, so the results are the
// bits of the unstaged one-lane kernel.
template <bool REDUCE, int ACC>
__global__ void __launch_bounds__(kStageBlock, 1)
plan_stage_kernel(const __grid_constant__ PlanParams p)
{
    const Terrain &T = p.T;
    const int n = T.ww * T.wh;
    for (int e = threadIdx.x; e < n; e += kStageBlock) {
        const int r = e / T.ww, c = e - r * T.ww;
        atp_win[e] = __ldg(T.tex + (size_t)(T.wy0 + r) * T.nx + (T.wx0 + c));
    }
    __syncthreads();
    const long long tid = (long long)blockIdx.x * kStageBlock + threadIdx.x;
    const int j = (int)tid;
    const bool live = tid < p.N;
    float J = 0.f, margin = CUDART_INF_F;
    bool feasible = false;
    if (live) rollout_one<false, TEX_F32W, ACC>(p, j, J, margin, feasible);
    if (!REDUCE) return;
    plan_tail<kStageBlock>(p, j, live, J, feasible, gridDim.x);
}

template <bool REDUCE, int ACC>
static cudaError_t launch_stage(const PlanParams &p, cudaStream_t stream)
{
    const size_t smem = (size_t)p.T.ww * p.T.wh * sizeof(float4);
    cudaError_t e = cudaFuncSetAttribute(plan_stage_kernel<REDUCE, ACC>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)(((size_t)p.N + kStageBlock - 1) / kStageBlock));
    plan_stage_kernel<REDUCE, ACC><<<grid, kStageBlock, smem, stream>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_plan_staged(const PlanParams &p, bool reduce, cudaStream_t stream)
{
    if (p.tex_format != TEX_F32W || p.x0_soa || p.T.ww < 2 || p.T.wh < 2 || p.T.ww > kStageMaxSide ||
        p.T.wh > kStageMaxSide || p.T.wx0 < 0 || p.T.wy0 < 0 || p.T.wx0 + p.T.ww > p.T.nx ||
        p.T.wy0 + p.T.wh > p.T.ny)
        return cudaErrorInvalidValue;
    if (reduce) return p.acc64 ? launch_stage<true, kAccF64>(p, stream) : launch_stage<true, kAccF32>(p, stream);
    return p.acc64 ? launch_stage<false, kAccF64>(p, stream) : launch_stage<false, kAccF32>(p, stream);
}

// Continuous batching: one launch over a ragged batch of plans, each with its
// own vehicle, terrain, horizon, candidates and outputs.  Plan r owns CTAs
// [cta_begin[r], cta_begin[r+1]) in the layout p.lanes, which the host chooses
// for the batch as a whole (every layout gives the same bits).  Every
// candidate runs exactly the code of a single plan, so its results are the
// same bits alone and in any mix.  BTEX is the batch's texel format when all
// its plans share one, or kTexMixed, where each plan branches on its own.
constexpr int kTexMixed = -1;

template <bool PER_X0, int TEX>
__device__ __forceinline__ bool batch_rollout(const PlanParams &p, void *sh, unsigned cta, int &j, float &J,
                                              float &margin, bool &feasible)
{
    // every thread of a CTA belongs to one plan: the branches are CTA-uniform
    if (p.lanes == kLayoutDuo4)
        return duo_rollout<4, PER_X0, TEX, kAccRuntime>(p, NoTrace{}, *(Duo<4> *)sh, cta, j, J, margin, feasible);
    if (p.lanes == kLayoutDuo2)
        return duo_rollout<2, PER_X0, TEX, kAccRuntime>(p, NoTrace{}, *(Duo<2> *)sh, cta, j, J, margin, feasible);
    if (p.lanes == kLayoutDuo1)
        return duo_rollout<1, PER_X0, TEX, kAccRuntime>(p, NoTrace{}, *(Duo<1> *)sh, cta, j, J, margin, feasible);
    j = (int)(cta * kPlanBlock + threadIdx.x);
    const bool live = j < p.N;
    if (live) rollout_one<PER_X0, TEX, kAccRuntime>(p, j, J, margin, feasible);
    return live;
}

template <int TEX>
__device__ __forceinline__ bool batch_tex(const PlanParams &p, void *sh, unsigned cta, int &j, float &J,
                                          float &margin, bool &feasible)
{
    return p.x0_soa ? batch_rollout<true, TEX>(p, sh, cta, j, J, margin, feasible)
                    : batch_rollout<false, TEX>(p, sh, cta, j, J, margin, feasible);
}

template <int BTEX>
__global__ void __launch_bounds__(kPlanBlock, 6)
plan_batch_kernel(const __grid_constant__ BatchParams b)
{
    __shared__ __align__(16) unsigned char sh[sizeof(Duo<1>)];
    static_assert(sizeof(Duo<1>) >= sizeof(Duo<2>) && sizeof(Duo<1>) >= sizeof(Duo<4>), "one buffer for all");
    int lo = 0, hi = b.n;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (b.cta_begin[mid] <= (int)blockIdx.x) lo = mid;
        else hi = mid;
    }
    const PlanParams &p = b.req[lo];
    const unsigned cta = blockIdx.x - (unsigned)b.cta_begin[lo];
    int j;
    float J = 0.f, margin = CUDART_INF_F;
    bool feasible = false, leader;
    if (BTEX == TEX_F32 || (BTEX == kTexMixed && p.tex_format == TEX_F32))
        leader = batch_tex<TEX_F32>(p, sh, cta, j, J, margin, feasible);
    else
        leader = batch_tex<TEX_BF16>(p, sh, cta, j, J, margin, feasible);
    plan_tail(p, j, leader, J, feasible, (unsigned)(b.cta_begin[lo + 1] - b.cta_begin[lo]));
}

cudaError_t launch_plan_batch(const BatchParams &b, cudaStream_t stream)
{
    if (b.n < 1 || b.n > kMaxBatch) return cudaErrorInvalidValue;
    bool f32 = true, bf16 = true;
    for (int r = 0; r < b.n; ++r) {
        f32 = f32 && b.req[r].tex_format == TEX_F32;
        bf16 = bf16 && b.req[r].tex_format == TEX_BF16;
    }
    const unsigned grid = (unsigned)b.cta_begin[b.n];
    if (f32) plan_batch_kernel<TEX_F32><<<grid, kPlanBlock, 0, stream>>>(b);
    else if (bf16) plan_batch_kernel<TEX_BF16><<<grid, kPlanBlock, 0, stream>>>(b);
    else plan_batch_kernel<kTexMixed><<<grid, kPlanBlock, 0, stream>>>(b);
    return cudaGetLastError();
}

template <bool PER_X0, bool REDUCE, int TEX, int ACC>
static void launch_layout(const PlanParams &p, int layout, cudaStream_t stream)
{
    const dim3 grid((unsigned)layout_ctas(layout, p.N)), block(kPlanBlock);
    if (layout == kLayoutDuo4) plan_duo_kernel<4, PER_X0, REDUCE, TEX, ACC><<<grid, block, 0, stream>>>(p);
    else if (layout == kLayoutDuo2) plan_duo_kernel<2, PER_X0, REDUCE, TEX, ACC><<<grid, block, 0, stream>>>(p);
    else if (layout == kLayoutDuo1) plan_duo_kernel<1, PER_X0, REDUCE, TEX, ACC><<<grid, block, 0, stream>>>(p);
    else plan_kernel<PER_X0, REDUCE, TEX, ACC><<<grid, block, 0, stream>>>(p);
}

template <int TEX, int ACC>
static cudaError_t launch_acc(const PlanParams &p, bool reduce, cudaStream_t stream)
{
    const int layout = plan_layout(p.lanes, p.N);
    if (reduce) {
        if (p.x0_soa) launch_layout<true, true, TEX, ACC>(p, layout, stream);
        else launch_layout<false, true, TEX, ACC>(p, layout, stream);
    } else {
        if (p.x0_soa) launch_layout<true, false, TEX, ACC>(p, layout, stream);
        else launch_layout<false, false, TEX, ACC>(p, layout, stream);
    }
    return cudaGetLastError();
}

cudaError_t launch_plan(const PlanParams &p, bool reduce, cudaStream_t stream)
{
    if (p.tex_format == TEX_F32)
        return p.acc64 ? launch_acc<TEX_F32, kAccF64>(p, reduce, stream) : launch_acc<TEX_F32, kAccF32>(p, reduce, stream);
    return p.acc64 ? launch_acc<TEX_BF16, kAccF64>(p, reduce, stream) : launch_acc<TEX_BF16, kAccF32>(p, reduce, stream);
}

// Texels (Sec. III-A numeric slope, reading Q10): height, central-difference
// slopes (one-sided on the border) and the costmap value per node.  Each
// thread makes kPrepRows nodes of a column, so that its loads overlap (one node
// per thread waited on them: 28 us for 2048^2 nodes against a 15 us floor of
// bytes) and neighbouring rows come from registers.
constexpr int kPrepRows = 4;

struct PrepNode {
    float c, gx, gy, cost;
};

// nodes (i, j0 .. j0 + kPrepRows - 1); rows beyond the map repeat the last
__device__ __forceinline__ void prep_column(const float *__restrict__ H, const float *__restrict__ cm, int nx, int ny,
                                            float inv_cell, int i, int j0, PrepNode (&n)[kPrepRows])
{
    const int il = i > 0 ? i - 1 : 0, ir = i < nx - 1 ? i + 1 : nx - 1;
    const float wx = i == 0 || i == nx - 1 ? inv_cell : 0.5f * inv_cell;
    float col[kPrepRows + 2], l[kPrepRows], r[kPrepRows];
#pragma unroll
    for (int q = 0; q < kPrepRows + 2; ++q)
        col[q] = __ldg(H + (size_t)min(max(j0 + q - 1, 0), ny - 1) * nx + i);
#pragma unroll
    for (int q = 0; q < kPrepRows; ++q) {
        const size_t o = (size_t)min(j0 + q, ny - 1) * nx;
        l[q] = __ldg(H + o + il);
        r[q] = __ldg(H + o + ir);
        n[q].cost = cm ? __ldg(cm + o + i) : 0.f;
    }
#pragma unroll
    for (int q = 0; q < kPrepRows; ++q) {
        const int j = j0 + q;
        n[q].c = col[q + 1];
        n[q].gx = (r[q] - l[q]) * wx;
        n[q].gy = (col[q + 2] - col[q]) * (j == 0 || j >= ny - 1 ? inv_cell : 0.5f * inv_cell);
    }
}

__global__ void __launch_bounds__(256) terrain_prepare_f32_kernel(const float *__restrict__ H,
                                                                  const float *__restrict__ cm, int nx, int ny,
                                                                  float inv_cell, float4 *__restrict__ out)
{
    const int i = blockIdx.x * 32 + threadIdx.x;
    const int j0 = (blockIdx.y * 8 + threadIdx.y) * kPrepRows;
    if (i >= nx || j0 >= ny) return;
    PrepNode n[kPrepRows];
    prep_column(H, cm, nx, ny, inv_cell, i, j0, n);
#pragma unroll
    for (int q = 0; q < kPrepRows; ++q)
        if (j0 + q < ny) out[(size_t)(j0 + q) * nx + i] = make_float4(n[q].c, n[q].gx, n[q].gy, n[q].cost);
}

__device__ __forceinline__ unsigned bf16_bits(float v)
{
    return (unsigned)__bfloat16_as_ushort(__float2bfloat16_rn(v));
}

// BF16 texels.  Per 8 x 8 block a plane through the block's first node with
// the slopes of its first row and first column (FP32, each operation rounded
// on its own so that the plane is reproducible bit for bit); per node the
// bf16 (round to nearest even) of the height's and the two node slopes'
// residuals from that plane, and of the costmap value.  Every thread forms
// its block's plane itself (three loads its warp shares), the block's first
// node stores it.
__global__ void __launch_bounds__(256) terrain_prepare_bf16_kernel(const float *__restrict__ H,
                                                                   const float *__restrict__ cm, int nx, int ny,
                                                                   float inv_cell, float4 *__restrict__ plane, int nbx,
                                                                   uint2 *__restrict__ out)
{
    const int i = blockIdx.x * 32 + threadIdx.x;
    const int j0 = (blockIdx.y * 8 + threadIdx.y) * kPrepRows;
    if (i >= nx || j0 >= ny) return;
    static_assert(8 % kPrepRows == 0, "a thread's nodes lie in one block");
    PrepNode n[kPrepRows];
    prep_column(H, cm, nx, ny, inv_cell, i, j0, n);
    const int bi = i & ~7, bj = j0 & ~7;
    const int ni = min(8, nx - bi), nj = min(8, ny - bj);
    const float c0 = __ldg(H + (size_t)bj * nx + bi);
    const float cx = ni > 1 ? __fmul_rn(__fsub_rn(__ldg(H + (size_t)bj * nx + bi + ni - 1), c0),
                                        __fdiv_rn(1.0f, (float)(ni - 1))) : 0.f;
    const float cy = nj > 1 ? __fmul_rn(__fsub_rn(__ldg(H + (size_t)(bj + nj - 1) * nx + bi), c0),
                                        __fdiv_rn(1.0f, (float)(nj - 1))) : 0.f;
    const float4 P = make_float4(c0, cx, cy, 0.f);
    if (i == bi && j0 == bj) plane[(size_t)(bj >> 3) * nbx + (bi >> 3)] = P;
#pragma unroll
    for (int q = 0; q < kPrepRows; ++q) {
        const int j = j0 + q;
        if (j >= ny) break;
        const float res = __fsub_rn(n[q].c, block_plane(P, i, j));
        // slopes as residuals from the plane's own slopes
        const float rgx = __fsub_rn(n[q].gx, __fmul_rn(P.y, inv_cell));
        const float rgy = __fsub_rn(n[q].gy, __fmul_rn(P.z, inv_cell));
        out[(size_t)j * nx + i] = make_uint2(bf16_bits(res) | (bf16_bits(rgx) << 16),
                                             bf16_bits(rgy) | (bf16_bits(n[q].cost) << 16));
    }
}

static dim3 prep_grid(int nx, int ny)
{
    return dim3((unsigned)((nx + 31) / 32), (unsigned)((ny + 8 * kPrepRows - 1) / (8 * kPrepRows)));
}

cudaError_t launch_terrain_prepare_bf16(const float *heights, const float *costmap, int nx, int ny,
                                        float inv_cell, uint2 *texels, float4 *plane, cudaStream_t stream)
{
    terrain_prepare_bf16_kernel<<<prep_grid(nx, ny), dim3(32, 8), 0, stream>>>(heights, costmap, nx, ny, inv_cell,
                                                                               plane, (nx + 7) / 8, texels);
    return cudaGetLastError();
}

cudaError_t launch_terrain_prepare_f32(const float *heights, const float *costmap, int nx, int ny,
                                       float inv_cell, float4 *out, cudaStream_t stream)
{
    terrain_prepare_f32_kernel<<<prep_grid(nx, ny), dim3(32, 8), 0, stream>>>(heights, costmap, nx, ny, inv_cell, out);
    return cudaGetLastError();
}

}  // namespace atp
