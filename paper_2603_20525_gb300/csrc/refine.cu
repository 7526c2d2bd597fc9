// refine.cu - projected-gradient refinement of candidate control sequences
// with the adjoint's gradient (atp_grad): the step arithmetic of one
// iteration.  K is small (the refined candidates are the best few of a plan),
// so the threads spread over the control steps too: one thread per candidate
// waited on one step's loads after another (24 us a trial and 21 us an accept
// for 64 candidates of 50 steps).  Layouts as the plan kernel's: ctrl, grad
// [H][K][2] (steering rate, acceleration), cost and step size [K].
#include <cuda_runtime.h>

#include "refine.cuh"

namespace atp {

namespace {

constexpr int kCands = 32, kSteps = 16;      // a CTA's candidates and step rows

// eta[j] = step / (max over k, c of |grad[k][j][c]| + 1e-12)
__global__ void __launch_bounds__(kCands * kSteps)
refine_init_kernel(const float2 *__restrict__ grad, int K, int H, float step, float *__restrict__ eta)
{
    __shared__ float s_m[kSteps][kCands];
    const int j = blockIdx.x * kCands + threadIdx.x;
    float m = 0.f;
    if (j < K) {
        for (int k = threadIdx.y; k < H; k += kSteps) {
            const float2 g = grad[(size_t)k * K + j];
            m = fmaxf(m, fmaxf(fabsf(g.x), fabsf(g.y)));
        }
    }
    s_m[threadIdx.y][threadIdx.x] = m;
    __syncthreads();
    if (threadIdx.y > 0 || j >= K) return;
#pragma unroll
    for (int q = 1; q < kSteps; ++q) m = fmaxf(m, s_m[q][threadIdx.x]);
    eta[j] = step / (m + 1e-12f);
}

// trial = ctrl - eta[j] grad, the steering rate projected onto its limit
// (the admissible set of Sec. IV-C)
__global__ void __launch_bounds__(kCands * kSteps)
refine_trial_kernel(const float2 *__restrict__ ctrl, const float2 *__restrict__ grad,
                    const float *__restrict__ eta, int K, int H, float rate_max, float2 *__restrict__ trial)
{
    const int j = blockIdx.x * kCands + threadIdx.x;
    if (j >= K) return;
    const float e = eta[j];
    for (int k = blockIdx.y * kSteps + threadIdx.y; k < H; k += gridDim.y * kSteps) {
        const size_t i = (size_t)k * K + j;
        const float2 u = ctrl[i], g = grad[i];
        float r = fmaf(-e, g.x, u.x);
        r = fminf(fmaxf(r, -rate_max), rate_max);
        trial[i] = make_float2(r, fmaf(-e, g.y, u.y));
    }
}

// accept the trial of candidate j where its cost is finite and lower: the
// controls, gradient and cost become the trial's and the step grows by 1.5;
// otherwise the step halves.  A candidate's steps lie in one CTA, which has
// read its old cost before it writes the new one.
__global__ void __launch_bounds__(kCands * kSteps)
refine_accept_kernel(int K, int H, const float2 *__restrict__ trial, const float *__restrict__ trial_cost,
                     const float2 *__restrict__ trial_grad, float2 *__restrict__ ctrl, float *__restrict__ cost,
                     float2 *__restrict__ grad, float *__restrict__ eta)
{
    const int j = blockIdx.x * kCands + threadIdx.x;
    const bool live = j < K;
    const float Jt = live ? trial_cost[j] : 0.f;
    const bool ok = live && isfinite(Jt) && Jt < cost[j];
    __syncthreads();
    if (!live) return;
    if (ok) {
        for (int k = threadIdx.y; k < H; k += kSteps) {
            const size_t i = (size_t)k * K + j;
            ctrl[i] = trial[i];
            grad[i] = trial_grad[i];
        }
    }
    if (threadIdx.y == 0) {
        if (ok) cost[j] = Jt;
        eta[j] *= ok ? 1.5f : 0.5f;
    }
}

unsigned blocks(int K) { return (unsigned)(((long long)K + kCands - 1) / kCands); }

}  // namespace

cudaError_t launch_refine_init(const float *grad, int K, int H, float step, float *eta, cudaStream_t stream)
{
    refine_init_kernel<<<blocks(K), dim3(kCands, kSteps), 0, stream>>>((const float2 *)grad, K, H, step, eta);
    return cudaGetLastError();
}

cudaError_t launch_refine_trial(const float *ctrl, const float *grad, const float *eta, int K, int H,
                                float rate_max, float *trial, cudaStream_t stream)
{
    const dim3 grid(blocks(K), (unsigned)(H < 64 * kSteps ? (H + kSteps - 1) / kSteps : 64));
    refine_trial_kernel<<<grid, dim3(kCands, kSteps), 0, stream>>>((const float2 *)ctrl, (const float2 *)grad, eta, K, H,
                                                          rate_max, (float2 *)trial);
    return cudaGetLastError();
}

cudaError_t launch_refine_accept(int K, int H, const float *trial, const float *trial_cost, const float *trial_grad,
                                 float *ctrl, float *cost, float *grad, float *eta, cudaStream_t stream)
{
    refine_accept_kernel<<<blocks(K), dim3(kCands, kSteps), 0, stream>>>(K, H, (const float2 *)trial, trial_cost,
                                                           (const float2 *)trial_grad, (float2 *)ctrl, cost,
                                                           (float2 *)grad, eta);
    return cudaGetLastError();
}

}  // namespace atp
