// The shadow splat's backward (shadow_bwd.cu), called by backward.cu.
#pragma once
#include "gs3_internal.cuh"

namespace gs3 {

struct ShadowBwdArgs {
  const float* dT;    // dL/dT by Gaussian index
  float2* ct;         // [N] scratch
  uint32_t* ticket;   // [4] zero: three tickets, and whether a coefficient is infinite or not a number
  float* light_geom;  // [N][8], zero: dL/dgamma, then the sums of w dx, w dy, w dx dy, w dx^2, w dy^2 over the
                      // light's pixels, w = dL/dpower and (dx, dy) = pixel - centre
  cudaEvent_t fork;   // records the point of `s` from which `side` may go on (side != s)
};
// Adds the shadow splat's gradients to light_geom: the open segments on `s`,
// the receivers of the stopped ones on `side` (which joins nothing).
void launch_shadow_backward(const FrameArgs& f, const ShadowBwdArgs& a, cudaStream_t s, cudaStream_t side);

}  // namespace gs3
