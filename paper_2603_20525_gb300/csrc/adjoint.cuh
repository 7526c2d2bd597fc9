// adjoint.cuh - parameters of the rollout-cost adjoint kernels.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>

namespace atp {

struct PlanParams;

// what the adjoint differentiates
constexpr int kGradCost = 0, kGradMargin = 1;

// Device memory of one adjoint call.  A trace (one record of 64 bytes per
// candidate and Euler step) of up to kTraceBytes is kept whole; a longer one
// is recomputed in segments of `seg` control steps from checkpoints.
constexpr size_t kTraceBytes = (size_t)1 << 30;
struct GradPlan {
    int seg, n_seg;                       // control steps per segment, segments
    size_t rec, ckpt, fin, lam, ints, total;   // byte offsets and size
};
GradPlan grad_plan(int K, int H, int n_sub, int ckpt);

// `p` holds the problem (p.N = K, p.cost the objective's value [K]); grad is
// [H][K][2] and buf grad_plan(...).total bytes.
cudaError_t launch_grad(const PlanParams &p, const GradPlan &g, int objective, char *buf, float *grad,
                        cudaStream_t stream);

}  // namespace atp
