// Residual kernels of the 2D problems; in FP64 the element arithmetic runs in
// 64-bit fixed point (fx64.cuh).
//
// A warp owns a strip of 30 node columns and marches along y on its own: lane l
// holds node column x0 + l, forms its w = x + eps v once a row, takes the right
// corners of element column x0 + l and the contributions of column x0 + l - 1
// from its neighbour lanes, and carries a row's contributions to the row above
// in registers.  No shared memory and no barrier, so small grids spread over
// the SMs a row or two a warp.
//
// Bound by the latency of a row's arithmetic on small grids and by instruction
// issue on large ones.  Measured against the FP64-pipe kernel (row segments of
// up to 512 columns marching 4 rows or more, FP64 exponentials): Bratu residual
// 33^2 22.5 -> 7.3 us; the FP64 65^2 Bratu solve 18.6 -> 8.2 ms; the 64-instance
// batched solve 172 -> 141 ms.
#pragma once
#include "element.cuh"
#include "fx64.cuh"
#include "stencil.cuh"
#include "stencil_body.cuh"

namespace jfnk {

constexpr int kFx2Strip = 30;     // node columns a warp completes
constexpr int kFx2Warps = 4;      // per CTA
// warps a launch is cut into, about what is resident: FP64 96 registers a thread
constexpr int kFx2Slots64 = kNumSMs * 20, kFx2Slots32 = kNumSMs * 40;

__host__ __device__ inline int fx2d_strips(int n) { return (n - 1 + kFx2Strip - 1) / kFx2Strip; }

// True when the kernels take this call: outputs apart from the vectors whose
// neighbouring values other lanes still read, (FP64) no node factor, and no more
// strips (a CTA has one) than the reduction scratch holds partials where the
// call reduces: n <= 61441, the row-segment kernel beyond.
template <typename T>
bool fx2d_use(Prob prob, const StencilArgs<T>& a, Mode mode);

template <typename T>
jfnk_status launch_fx2d(Prob prob, Mode mode, const StencilArgs<T>& a, cudaStream_t st);

#ifdef __CUDACC__

// FP64 evaluation of element (x, y), for values outside the fixed-point range.
template <Prob P, bool JV>
__device__ __noinline__ void elem2_fp64(const StencilArgs<double>& a, double eps, int x, int y, double* r) {
    const int n = a.g.n;
    double w[4];
    for (int c = 0; c < 4; ++c) {
        const int X = x + (c & 1), Y = y + (c >> 1);
        const long long i = JFNK_IDX((long long)Y * a.g.sy + X, a.g.size);
        const bool bnd = X == 0 || X == n || Y == 0 || Y == n;
        w[c] = a.u[i];
        if (JV && !bnd) w[c] = fma(eps, a.v[i], w[c]);
    }
    if (P == Prob::MINSURF2)
        elem_minsurf2<double>(w, a.lh, r);
    else
        elem_bratu2<double>(w, a.lh, r);
}

// Node rows [y0, y1) of a strip, by one warp.
template <Prob P, Mode M>
__device__ __forceinline__ void fx2d_warp(const StencilArgs<double>& a, int strip, int y0, int y1, float& red) {
    const unsigned int all = 0xffffffffu;
    const int n = a.g.n;
    const int lane = threadIdx.x & 31;
    const int x = strip * kFx2Strip + lane;
    const bool col = x <= n;                              // a node column of the grid
    const bool elem_x = x < n && lane < 31;               // lane 31 only lends its node to element 30
    const bool inner_x = x > 0 && x < n;
    const bool out_x = col && (lane == 0 ? x == 0 : lane < 31 || x == n);
    double eps = 0.0, inv_eps = 0.0;
    if (M != Mode::F) {
        eps = eps_of<double>(a.eps);
        inv_eps = inv_eps_of<double>(a.eps);
    }
    ChebK<double> ck = {0.0, 0.0, 0.0};
    if (M == Mode::CHEB0 || M == Mode::CHEB || M == Mode::CHEBLAST) ck = cheb_of<double>(a.cheb, a.cheb_step);
    const bool par_ok = P == Prob::MINSURF2 ? fx_scale_ok(a.lh) : fx_bratu_ok(a.lh);
    FxBratu br;
    FxMinsurf mi;
    if (P == Prob::MINSURF2)
        mi = fx_minsurf(par_ok ? a.lh : 1.0);
    else
        br = fx_bratu(par_ok ? a.lh : 0.0);

    double ru = 0.0, rv = 0.0;
    auto fetch = [&](int y) {
        if (!col || y < 0 || y > n) return;
        const long long i = JFNK_IDX((long long)y * a.g.sy + x, a.g.size);
        ru = a.u[i];
        if (M != Mode::F) rv = (inner_x && y > 0 && y < n) ? a.v[i] : 0.0;
    };
    fx_t p[4] = {0, 0, 0, 0}, carry[2] = {0, 0};  // corners; contributions to the upper row ...
    int Xc = kFxTiny;                             // ... times 2^Xc, or doubles (kFxFp64)
    auto row = [&](fx_t* q) {                     // the fetched row's values of this column and the next
        q[0] = col ? fx_pack(M != Mode::F ? fma(eps, rv, ru) : ru) : 0;
        q[1] = __shfl_down_sync(all, q[0], 1);
    };
    fetch(y0 - 1);
    if (y0 > 0) row(p);
    fetch(y0);
    for (int j = y0 - 1; j < y1; ++j) {
        row(p + 2);
        fetch(j + 2);
        const bool out = out_x && j >= y0, inner = out && inner_x && j > 0 && j < n;
        const long long idx = (long long)j * a.g.sy + x;
        EpiIn1<double> e;
        if (inner) epi1_load<double, M>(a, idx, e);
        fx_t r[4] = {0, 0, 0, 0};
        int Xr = kFxTiny;
        if (elem_x && j >= 0 && j < n) {
            const int xm = max(max(fx_exp(p[0]), fx_exp(p[1])), max(fx_exp(p[2]), fx_exp(p[3])));
            bool done;
            if (P == Prob::MINSURF2) {
                done = xm == 0;
                if (par_ok && fx_exp_ok(xm)) done = fx_minsurf2(p, xm, mi, r, Xr);
                if (!done) Xr = kFxTiny;
            } else {
                // a zero element: the source alone (its exponent is any)
                const int xe = xm == 0 ? kFxMinExp : xm;
                done = par_ok && fx_bratu_exp_ok(xe);
                if (done) fx_bratu2(p, xe, br, r, Xr);
            }
            if (!done) {
                double rs[4];
                elem2_fp64<P, M != Mode::F>(a, eps, x, j, rs);
#pragma unroll
                for (int c = 0; c < 4; ++c) r[c] = __double_as_longlong(rs[c]);
                Xr = kFxFp64;
            }
        }
        // node row j: this element row's lower contributions and the carried ones
        double d[2];
        if (Xr != kFxFp64 && Xc != kFxFp64) {
            const int X = max(Xr, Xc) + 1;  // (one bit of room for the sum)
#pragma unroll
            for (int c = 0; c < 2; ++c) d[c] = fx_to_double(fx_sar(carry[c], X - Xc) + fx_sar(r[c], X - Xr), X);
        } else {
#pragma unroll
            for (int c = 0; c < 2; ++c)
                d[c] = (Xc == kFxFp64 ? __longlong_as_double(carry[c]) : fx_to_double(carry[c], Xc)) +
                       (Xr == kFxFp64 ? __longlong_as_double(r[c]) : fx_to_double(r[c], Xr));
        }
        const double left = __shfl_up_sync(all, d[1], 1);
        if (inner)
            epilogue_pf<double, M>(a, idx, true, left + d[0], inv_eps, ck, e, red);
        else if (out)
            epilogue<double, M>(a, idx, false, 0.0, 0.0, ck, red);  // Dirichlet nodes: zero
        carry[0] = r[2];
        carry[1] = r[3];
        Xc = Xr;
        p[0] = p[2];
        p[1] = p[3];
    }
}

// The same in FP32, element arithmetic in FP32.  Bound by instruction
// issue: 146 instructions an element at 67 % of the issue slots on 4097^2 nodes
// (fetching rows 2 to 4 ahead instead of 1 changed nothing).  Residual against
// the row-segment kernel: 1025^2 14.5 -> 10.3 us, 2049^2 37.1 -> 25.0 us, 4097^2
// 127 -> 101 us.
template <Prob P, Mode M>
__device__ __forceinline__ void fx2d_warp(const StencilArgs<float>& a, int strip, int y0, int y1, float& red) {
    const unsigned int all = 0xffffffffu;
    const int n = a.g.n;
    const int lane = threadIdx.x & 31;
    const int x = strip * kFx2Strip + lane;
    const bool col = x <= n;
    const bool inner_x = x > 0 && x < n;
    const bool out_x = col && (lane == 0 ? x == 0 : lane < 31 || x == n);
    float eps = 0.f, inv_eps = 0.f;
    if (M != Mode::F) {
        eps = eps_of<float>(a.eps);
        inv_eps = inv_eps_of<float>(a.eps);
    }
    ChebK<float> ck = {0.f, 0.f, 0.f};
    if (M == Mode::CHEB0 || M == Mode::CHEB || M == Mode::CHEBLAST) ck = cheb_of<float>(a.cheb, a.cheb_step);
    float ru = 0.f, rv = 0.f;
    auto fetch = [&](int y) {
        if (!col || y < 0 || y > n) return;
        const long long i = JFNK_IDX((long long)y * a.g.sy + x, a.g.size);
        ru = a.u[i];
        if (M != Mode::F) rv = (inner_x && y > 0 && y < n) ? a.v[i] : 0.f;
    };
    float p[4] = {0.f, 0.f, 0.f, 0.f}, carry[2] = {0.f, 0.f};
    auto row = [&](float* q) {
        q[0] = M != Mode::F ? ru + eps * rv : ru;
        q[1] = __shfl_down_sync(all, q[0], 1);
    };
    fetch(y0 - 1);
    row(p);
    fetch(y0);
    for (int j = y0 - 1; j < y1; ++j) {
        row(p + 2);
        fetch(j + 2);
        const bool out = out_x && j >= y0, inner = out && inner_x && j > 0 && j < n;
        const long long idx = (long long)j * a.g.sy + x;
        EpiIn1<float> e;
        if (inner) epi1_load<float, M>(a, idx, e);
        float r[4];
        if (P == Prob::MINSURF2)
            elem_minsurf2<float>(p, a.lh, r);
        else
            elem_bratu2<float>(p, a.lh, r);
        // (rows and columns outside the grid only feed nodes that are not inner)
        const float left = __shfl_up_sync(all, carry[1] + r[1], 1);
        if (inner)
            epilogue_pf<float, M>(a, idx, true, (left + (carry[0] + r[0])) * a.node_scale, inv_eps, ck, e, red);
        else if (out)
            epilogue<float, M>(a, idx, false, 0.f, 0.f, ck, red);
        carry[0] = r[2];
        carry[1] = r[3];
        p[0] = p[2];
        p[1] = p[3];
    }
}

// A CTA's part: node rows [y0, y1) of a strip, shared out among its warps.
template <Prob P, Mode M, typename T>
__device__ __forceinline__ void fx2d_cta(const StencilArgs<T>& a, int strip, int y0, int y1, unsigned int bid,
                                         unsigned int nb, double* red_sm) {
    const int warps = blockDim.x >> 5, w = threadIdx.x >> 5;
    const int per = (y1 - y0 + warps - 1) / warps;
    const int ya = y0 + w * per, yb = min(y1, ya + per);
    float red = 0.f;
    if (ya < yb) fx2d_warp<P, M>(a, strip, ya, yb, red);
    stencil_reduce(a, red, red_sm, bid, nb);
}
#endif

// Rows a CTA takes so that `rows` (strips x node rows, over all grids of a
// launch) fill the resident warps once.
inline int fx2d_cta_rows(long long rows, int slots, int warps = kFx2Warps) {
    const long long per = (rows + slots - 1) / slots;
    return warps * (int)(per < 1 ? 1 : per);
}

}  // namespace jfnk
