// FP32 kernels of the 3D diffusion problems: z-marching tiles, one launch per
// action, no scratch (stencil_t3.cu).
#pragma once
#include "stencil.cuh"

namespace jfnk {

// The tiling for a grid; no CTAs where the kernel does not apply.
FxTiling t3d_tiling(const Grid& g);

// True when the kernel takes this FP32 call: a.t3 is set, outputs apart from u
// and v, and no per-element output.
bool t3d_use(const StencilArgs<float>& a, Mode mode, bool adj);

jfnk_status launch_t3d(Prob prob, Mode mode, bool adj, const StencilArgs<float>& a, cudaStream_t st);

}  // namespace jfnk
