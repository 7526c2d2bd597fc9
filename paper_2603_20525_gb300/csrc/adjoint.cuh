// adjoint.cuh - parameters of the rollout-cost adjoint kernels.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>

namespace atp {

struct PlanParams;

// what the adjoint differentiates
constexpr int kGradCost = 0, kGradMargin = 1;

// Device memory of one adjoint call.  The trace (one record of 64 bytes per
// candidate and Euler step) is kept whole up to kWholeBytes (the L2), and
// beyond where the workspace that `ckpt` allows holds it (atp_grad in atp.h).
// Else it is recomputed in segments of `seg` control steps from checkpoints,
// and all but the last segment's share of the forward pass runs twice: 16384
// candidates of 400 steps take 1.85 ms with a whole trace and 2.05 ms in two
// segments, 65536 take 7.3 and 7.8 ms.
constexpr size_t kWholeBytes = (size_t)128 << 20, kTwoBytes = (size_t)16 << 30;
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
