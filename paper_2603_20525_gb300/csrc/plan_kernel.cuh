// plan_kernel.cuh - parameters and launchers of the fused rollout + argmin
// kernel (arxiv 2603.20525, Sec. IV-A..IV-D).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "atp.h"
#include "srb_model.cuh"

namespace atp {

// Reduction scratch of one plan: the packed argmin key, the feasible count and
// the ticket that elects the last CTA.  The last CTA restores the initial
// values, so consecutive plans on one stream need no memset.
struct Scratch {
    unsigned long long key;   // initial ~0ull
    unsigned int count;       // initial 0
    unsigned int ticket;      // initial 0
};

struct PlanParams {
    Veh V;
    Cost C;
    Terrain T;
    float x0[13];             // shared initial state (x0_soa == nullptr)
    const float *x0_soa;      // [13][N] per-candidate initial states, or nullptr
    const float2 *ctrl;       // [H][N]
    int N, H, n_sub;
    float h;                  // Euler step dt / n_sub
    float *cost;              // [N] or nullptr
    float *margin;            // [N] or nullptr
    uint8_t *flags;           // [N] or nullptr
    float *xf;                // [13][N] or nullptr
    float *step_margin;       // [H][N] or nullptr: each control step's minimum U_ESM
    int *min_step;            // [N] or nullptr: control step of each candidate's smallest
                              // per-step margin (the final state folded into step H-1)
    int tex_format;           // TEX_F32 or TEX_BF16
    int acc64;                // accumulate the running cost in FP64
    int lanes;                // 0: by batch size; else 1, 2 or 4 threads per candidate
                              // (in a batch: the layout)
    // plan only
    atp_plan_out *out;
    float *best_ctrl;         // [H][2] or nullptr
    float *best_margin;       // [H] or nullptr
    Scratch *scratch;
};

constexpr int kPlanBlock = 64;
// Layouts of a plan's CTAs of 64 threads, as threads per candidate: one
// thread, or two warps that share 32, 16 or 8 candidates (one, two or four
// lanes of each warp per candidate).  All give the same bits.
constexpr int kLayoutOne = 1, kLayoutDuo1 = 2, kLayoutDuo2 = 4, kLayoutDuo4 = 8;
// ms per plan on a GB300, scaled workload, H = 100, 4 Euler steps per control
// step, terrain seed 5:
//   candidates        8 threads   4 threads   2 threads   1 thread
//   1024                0.158       0.180       0.225       0.287
//   4096                0.176       0.182       0.232       0.297
//   4864                0.178       0.182       0.227       0.295
//   8192                0.242       0.216       0.231       0.299
//   12288               0.390       0.259       0.270       0.304
//   16384               0.424       0.315       0.284       0.305
//   20480               0.601       0.471       0.355       0.401
//   28672               0.698       0.508       0.371       0.410
//   32768               0.828       0.565       0.610       0.415
// 4864 = 152 x 4 x 8 candidates is four CTAs per SM on eight threads and 29184
// = 152 x 6 x 32 the one wave of six CTAs per SM on two; there the next layout
// becomes the faster one.  Four threads and two cross between 14336 candidates
// (means of five terrains each of three workloads, four against two: 0.279 /
// 0.303, 0.277 / 0.308 and 0.259 / 0.269 ms) and 16384 (0.327 / 0.314, 0.326 /
// 0.319, 0.309 / 0.277): up to 10 % is lost just below the line, where one
// workload's terrains spread more than that (0.285 to 0.369 ms on two).
constexpr int kDuo4MaxN = 4864;
constexpr int kDuo2MaxN = 16384;
constexpr int kDuo1MaxN = 29184;

// the layout of a plan of N candidates: `forced` (1, 2 or 4 threads per
// candidate) if set, else by batch size
inline int plan_layout(int forced, int N)
{
    static_assert(kLayoutOne == 1 && kLayoutDuo1 == 2 && kLayoutDuo2 == 4, "a layout is its threads");
    if (forced) return forced;
    return N <= kDuo4MaxN ? kLayoutDuo4 : N <= kDuo2MaxN ? kLayoutDuo2 : N <= kDuo1MaxN ? kLayoutDuo1 : kLayoutOne;
}
inline int layout_candidates(int layout) { return kPlanBlock / layout; }       // per CTA
inline long long layout_ctas(int layout, long long N)
{
    return (N + layout_candidates(layout) - 1) / layout_candidates(layout);
}
// threads per candidate as atp_plan_lanes counts them: 1, 2 or 4, where 4 may
// be eight
inline int plan_lanes(int forced, int N)
{
    const int l = plan_layout(forced, N);
    return l > 4 ? 4 : l;
}
cudaError_t launch_plan(const PlanParams &p, bool reduce, cudaStream_t stream);

// Terrain staging (one lane per candidate, F32 texels, a shared start
// state): CTAs of kStageBlock threads, each of which first copies the window
// p.T.(wx0, wy0, ww, wh) of the texel array into its shared memory.
constexpr int kStageBlock = 512;
constexpr int kStageMaxSide = 120;     // 120 x 120 texels = 225 KB
cudaError_t launch_plan_staged(const PlanParams &p, bool reduce, cudaStream_t stream);

// A ragged batch of plans in one launch.  The descriptors travel in the
// kernel's parameter block (at most 32 KB), so a batch needs no device copy.
constexpr int kMaxBatch = 64;
struct BatchParams {
    int n;
    int cta_begin[kMaxBatch + 1];   // CTA prefix: plan r owns [cta_begin[r], cta_begin[r+1])
    PlanParams req[kMaxBatch];
};
static_assert(sizeof(BatchParams) <= 32764, "batch descriptors exceed the kernel parameter limit");

cudaError_t launch_plan_batch(const BatchParams &b, cudaStream_t stream);
cudaError_t launch_terrain_prepare_f32(const float *heights, const float *costmap, int nx, int ny,
                                       float inv_cell, float4 *out, cudaStream_t stream);
cudaError_t launch_terrain_prepare_bf16(const float *heights, const float *costmap, int nx, int ny,
                                        float inv_cell, uint2 *texels, float4 *plane, cudaStream_t stream);

// byte offset of the BF16 block planes after the texels
inline size_t bf16_base_offset(int nx, int ny) { return ((size_t)nx * ny * 8 + 255) / 256 * 256; }

}  // namespace atp
