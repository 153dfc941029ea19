// Residual kernels of one 2D problem (their body is in stencil_fx2d.cuh;
// batch.cu runs it over a batch).
#include <algorithm>

#include "reduce.cuh"
#include "stencil_fx.cuh"
#include "stencil_fx2d.cuh"

namespace jfnk {

template <typename T, Prob P, Mode M>
__global__ void __launch_bounds__(32 * kFx2Warps) fx2d_kernel(const StencilArgs<T> a, int rows) {
    __shared__ double red_sm[32];
    const int y0 = blockIdx.y * rows;
    fx2d_cta<P, M>(a, blockIdx.x, y0, min(y0 + rows, a.g.ny), blockIdx.x + gridDim.x * blockIdx.y,
                   gridDim.x * gridDim.y, red_sm);
}

template <typename T>
bool fx2d_use(Prob prob, const StencilArgs<T>& a, Mode mode) {
    return is_2d(prob) && a.g.n >= 2 && (sizeof(T) == 4 || a.node_scale == T(1)) &&
           (a.red == RedOut::NONE || fx2d_strips(a.g.n) <= 2 * kMaxRedBlocks) && !fx_outputs_alias(a, mode);
}
template bool fx2d_use<double>(Prob, const StencilArgs<double>&, Mode);
template bool fx2d_use<float>(Prob, const StencilArgs<float>&, Mode);

template <typename T, Prob P, Mode M>
static jfnk_status launch_fx2d_pm(const StencilArgs<T>& a, cudaStream_t st) {
    const int strips = fx2d_strips(a.g.n);
    // (the reduction scratch holds 2 kMaxRedBlocks partials)
    int rows = fx2d_cta_rows((long long)strips * a.g.ny, sizeof(T) == 8 ? kFx2Slots64 : kFx2Slots32);
    const int most = std::max(1, 2 * kMaxRedBlocks / strips);
    rows = std::max(rows, (a.g.ny + most - 1) / most);
    fx2d_kernel<T, P, M><<<dim3(strips, (a.g.ny + rows - 1) / rows), 32 * kFx2Warps, 0, st>>>(a, rows);
    JFNK_LAUNCH_CHECK();
    return JFNK_OK;
}

template <typename T, Prob P>
static jfnk_status launch_fx2d_p(Mode mode, const StencilArgs<T>& a, cudaStream_t st) {
    switch (mode) {
        case Mode::F: return launch_fx2d_pm<T, P, Mode::F>(a, st);
        case Mode::JV: return launch_fx2d_pm<T, P, Mode::JV>(a, st);
        case Mode::BMJ: return launch_fx2d_pm<T, P, Mode::BMJ>(a, st);
        case Mode::CHEB0: return launch_fx2d_pm<T, P, Mode::CHEB0>(a, st);
        case Mode::CHEB: return launch_fx2d_pm<T, P, Mode::CHEB>(a, st);
        case Mode::CHEBLAST: return launch_fx2d_pm<T, P, Mode::CHEBLAST>(a, st);
    }
    set_error("unknown stencil mode");
    return JFNK_ERR_INVALID_ARG;
}

template <typename T>
jfnk_status launch_fx2d(Prob prob, Mode mode, const StencilArgs<T>& a, cudaStream_t st) {
    if (prob == Prob::MINSURF2) return launch_fx2d_p<T, Prob::MINSURF2>(mode, a, st);
    return launch_fx2d_p<T, Prob::BRATU2>(mode, a, st);
}
template jfnk_status launch_fx2d<double>(Prob, Mode, const StencilArgs<double>&, cudaStream_t);
template jfnk_status launch_fx2d<float>(Prob, Mode, const StencilArgs<float>&, cudaStream_t);

}  // namespace jfnk
