// FP64 kernels of the 3D diffusion problems with the element
// arithmetic in 64-bit fixed point (fx64.cuh): one launch per action, no
// scratch.
#pragma once
#include "stencil.cuh"

namespace jfnk {

// The tiling for a grid; no CTAs where the kernel does not apply (scalar 3D
// grids up to n = 1024 only).
FxTiling fx3d_tiling(const Grid& g);

// True when an output of the action overlaps u or v, whose neighbouring values
// the one-launch kernels still read while others write.
template <typename T>
bool fx_outputs_alias(const StencilArgs<T>& a, Mode mode);

// True when the fixed-point kernel takes this FP64 call: a.fx is set, and the
// outputs are apart from the vectors whose neighbouring values other threads
// still read.  adj: the vector-Jacobian product (not with the coefficient's
// derivative).
bool fx3d_use(const StencilArgs<double>& a, Mode mode, bool adj);

jfnk_status launch_fx3d(Prob prob, Mode mode, bool adj, const StencilArgs<double>& a, cudaStream_t st);

}  // namespace jfnk
