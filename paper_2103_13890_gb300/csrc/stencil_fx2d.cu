// FP64 residual of one 2D problem, element arithmetic in 64-bit fixed point
// (the kernel's body is in stencil_fx2d.cuh; batch.cu runs it over a batch).
#include <algorithm>

#include "reduce.cuh"
#include "stencil_fx.cuh"
#include "stencil_fx2d.cuh"

namespace jfnk {

template <Prob P, Mode M>
__global__ void __launch_bounds__(32 * kFx2Warps) fx2d_kernel(const StencilArgs<double> a, int rows) {
    __shared__ double red_sm[32];
    const int y0 = blockIdx.y * rows;
    fx2d_cta<P, M>(a, blockIdx.x, y0, min(y0 + rows, a.g.ny), blockIdx.x + gridDim.x * blockIdx.y,
                   gridDim.x * gridDim.y, red_sm);
}

bool fx2d_use(Prob prob, const StencilArgs<double>& a, Mode mode) {
    return is_2d(prob) && a.g.n >= 2 && a.node_scale == 1.0 && !fx_outputs_alias(a, mode);
}

template <Prob P, Mode M>
static jfnk_status launch_fx2d_pm(const StencilArgs<double>& a, cudaStream_t st) {
    const int strips = fx2d_strips(a.g.n);
    // (the reduction scratch holds 2 kMaxRedBlocks partials)
    int rows = fx2d_cta_rows((long long)strips * a.g.ny);
    const int most = std::max(1, 2 * kMaxRedBlocks / strips);
    rows = std::max(rows, (a.g.ny + most - 1) / most);
    fx2d_kernel<P, M><<<dim3(strips, (a.g.ny + rows - 1) / rows), 32 * kFx2Warps, 0, st>>>(a, rows);
    JFNK_LAUNCH_CHECK();
    return JFNK_OK;
}

template <Prob P>
static jfnk_status launch_fx2d_p(Mode mode, const StencilArgs<double>& a, cudaStream_t st) {
    switch (mode) {
        case Mode::F: return launch_fx2d_pm<P, Mode::F>(a, st);
        case Mode::JV: return launch_fx2d_pm<P, Mode::JV>(a, st);
        case Mode::BMJ: return launch_fx2d_pm<P, Mode::BMJ>(a, st);
        case Mode::CHEB0: return launch_fx2d_pm<P, Mode::CHEB0>(a, st);
        case Mode::CHEB: return launch_fx2d_pm<P, Mode::CHEB>(a, st);
        case Mode::CHEBLAST: return launch_fx2d_pm<P, Mode::CHEBLAST>(a, st);
    }
    set_error("unknown stencil mode");
    return JFNK_ERR_INVALID_ARG;
}

jfnk_status launch_fx2d(Prob prob, Mode mode, const StencilArgs<double>& a, cudaStream_t st) {
    if (prob == Prob::MINSURF2) return launch_fx2d_p<Prob::MINSURF2>(mode, a, st);
    return launch_fx2d_p<Prob::BRATU2>(mode, a, st);
}

}  // namespace jfnk
