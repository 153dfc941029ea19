// FP64 residual and vector-Jacobian product of the 3D diffusion problems, element
// arithmetic in 64-bit fixed point (fx64.cuh).
//
// One launch per action.  A CTA takes a tile of element columns and marches it
// along z; thread (tx, ty) evaluates one element per layer.  The values
// w = x + eps v of a node plane are formed once per tile and staged in shared
// memory; an element's contributions to its upper face stay in registers for
// the next layer, and those to the three columns beside it go through shared
// memory, so that each node sums its 8 contributions in a fixed order.  One
// barrier a layer: planes and contributions are double-buffered.
// Tiles overlap by one element in x and y (the nodes between two tiles need
// the elements of both sides), and a CTA's first layer only feeds the plane
// above it.  The (tile, plane) pairs are dealt to the CTAs in equal contiguous
// runs, so that the last wave is as full as the others.
//
// Bound by instruction issue and dependent chains of integer arithmetic (about
// 1200 instructions an element, 700 of them its arithmetic; half of the issue
// slots busy); measured against the FP64-pipe kernels
// (stencil_ep.cu): residual 129^3 0.622 -> 0.127 ms, 257^3 4.89 -> 0.844 ms, FD
// action with kappa 101^3 0.414 -> 0.075 ms.  CTAs of at most 288 threads, two
// per SM, 96 registers: 257^3 residual 0.844 ms, against 0.903 (576 x 1), 1.035
// (192 x 3) and 0.901 ms (256 x 2, 128 registers).
#include <algorithm>

#include "element.cuh"
#include "fx64.cuh"
#include "reduce.cuh"
#include "stencil.cuh"
#include "stencil_body.cuh"
#include "stencil_fx.cuh"

namespace jfnk {

constexpr int kFxThreads = 288, kFxBlocks = 2;  // largest CTA, CTAs per SM

// FP64 evaluation of the element at (x, y, z), for values outside the
// fixed-point range (non-finite or huge values, magnitudes near underflow,
// kappa <= 0).
template <bool KAPPA, bool JV>
__device__ __noinline__ void nd3_fp64(const StencilArgs<double>& a, double eps, int x, int y, int z, double kap,
                                      double* r) {
    const int n = a.g.n;
    double w[8];
    for (int c = 0; c < 8; ++c) {
        const int X = x + (c & 1), Y = y + ((c >> 1) & 1), Z = z + (c >> 2);
        const long long i = JFNK_IDX((long long)Z * a.g.sz + (long long)Y * a.g.sy + X, a.g.size);
        const bool bnd = X == 0 || X == n || Y == 0 || Y == n || Z == 0 || Z == n;
        w[c] = a.u[i];
        if (JV && !bnd) w[c] = fma(eps, a.v[i], w[c]);
    }
    elem_nd3<double, KAPPA>(w, kap, r);
    for (int c = 0; c < 8; ++c) r[c] *= a.node_scale;
}

// The same for the vector-Jacobian product, w = v at the unknowns.
template <bool KAPPA>
__device__ __noinline__ void vjp3_fp64(const StencilArgs<double>& a, int x, int y, int z, double kap, double* r) {
    const int n = a.g.n;
    double u[8], w[8], dk;
    for (int c = 0; c < 8; ++c) {
        const int X = x + (c & 1), Y = y + ((c >> 1) & 1), Z = z + (c >> 2);
        const long long i = JFNK_IDX((long long)Z * a.g.sz + (long long)Y * a.g.sy + X, a.g.size);
        const bool bnd = X == 0 || X == n || Y == 0 || Y == n || Z == 0 || Z == n;
        u[c] = a.u[i];
        w[c] = bnd ? 0.0 : a.v[i];
    }
    elem_vjp3<double>(u, w, kap, r, dk);
    for (int c = 0; c < 8; ++c) r[c] *= a.node_scale;
}

// ADJ: J^T v in place of the FD action; the planes of v are staged beside those
// of u.  About 1.8 times the instructions of a residual: 129^3 with kappa 0.228 ms
// against 1.068 ms of the FP64-pipe kernels, 257^3 1.54 against 8.43 ms.  (96
// registers spill some 20 values; one CTA an SM with 168 registers and none: 0.250
// and 1.78 ms.)
template <Prob P, Mode M, bool ADJ>
__global__ void __launch_bounds__(kFxThreads, kFxBlocks) fx3d_kernel(const StencilArgs<double> a) {
    const FxTiling& t = a.fx;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double red_sm[32];
    constexpr bool KAPPA = P == Prob::NDK3;
    const int n = a.g.n;
    const int sy = (int)a.g.sy, sz = (int)a.g.sz;
    const int npx = t.ex + 1, np = npx * (t.ey + 1), ne = t.ex * t.ey;
    fx_t* const W = reinterpret_cast<fx_t*>(smem_raw);        // [2][np] node planes, packed values
    fx_t* const V = W + (ADJ ? 2 * np : 0);                   // [2][np] those of the direction (ADJ)
    double* const C = reinterpret_cast<double*>(V + 2 * np);  // [2][3][ne] contributions to the neighbour columns
    const int tid = threadIdx.x;
    double eps = 0.0, inv_eps = 0.0;
    if (!ADJ && M != Mode::F) {
        eps = eps_of<double>(a.eps);
        inv_eps = inv_eps_of<double>(a.eps);
    }
    ChebK<double> ck = {0.0, 0.0, 0.0};
    if (M == Mode::CHEB0 || M == Mode::CHEB || M == Mode::CHEBLAST) ck = cheb_of<double>(a.cheb, a.cheb_step);
    const FxScale sc0 = fx_scale(a.node_scale);
    // this thread's node of a staged plane and element of a layer
    const int nx = tid % npx, ny = tid / npx;
    const int ex = tid % t.ex, ey = tid / t.ex;
    const int corner = ey * npx + ex;
    float red = 0.f;

    int step = (int)((long long)t.steps * blockIdx.x / gridDim.x);
    const int last = (int)((long long)t.steps * (blockIdx.x + 1) / gridDim.x);
    while (step < last) {
        const int tile = step / (n - 1);
        const int za = step - tile * (n - 1) + 1;         // first plane of this run
        const int zb = min(n, za + (last - step));        // one past its last
        step += zb - za;
        const int x0 = (tile % t.tx) * (t.ex - 1), y0 = (tile / t.tx) * (t.ey - 1);
        const int X = x0 + nx, Y = y0 + ny;
        const bool stage = tid < np && X <= n && Y <= n;
        const int sidx = Y * sy + X;
        const bool edge = X == 0 || X == n || Y == 0 || Y == n;
        const int gx = x0 + ex, gy = y0 + ey;
        const bool elem = tid < ne && gx < n && gy < n;
        const bool node = elem && ex > 0 && ey > 0;
        const int gidx = gy * sy + gx;
        const int eidx = gy * n + gx;

        double ru = 0.0, rv = 0.0;
        auto fetch = [&](int z) {
            if (!stage) return;
            const int i = (int)JFNK_IDX(z * sz + sidx, a.g.size);
            ru = a.u[i];
            if (M != Mode::F && !edge && z > 0 && z < n) rv = a.v[i]; else rv = 0.0;
        };
        auto store = [&](int z) {
            if (!stage) return;
            W[(z & 1) * np + tid] = fx_pack(!ADJ && M != Mode::F ? fma(eps, rv, ru) : ru);
            if (ADJ) V[(z & 1) * np + tid] = fx_pack(rv);
            // Dirichlet nodes: every output is zero
            if (edge || z == 0 || z == n) {
                if (ADJ)
                    epilogue_adj<double, M>(a, z * sz + sidx, false, 0.0, ck, red);
                else
                    epilogue<double, M>(a, z * sz + sidx, false, 0.0, 0.0, ck, red);
            }
        };
        fx_t p[8], pv[ADJ ? 8 : 1], carry[4] = {0, 0, 0, 0};  // corners; contributions to the upper face ...
        int xl = 0, xvl = 0, Xc = kFxTiny;   // ... times 2^Xc, or doubles (kFxFp64)
        auto face = [&](const fx_t* plane, int z, fx_t* q) -> int {
            const fx_t* Wz = plane + (z & 1) * np + corner;
            q[0] = Wz[0];
            q[1] = Wz[1];
            q[2] = Wz[npx];
            q[3] = Wz[npx + 1];
            return max(max(fx_exp(q[0]), fx_exp(q[1])), max(fx_exp(q[2]), fx_exp(q[3])));
        };
        fetch(za - 1);
        store(za - 1);
        fetch(za);
        store(za);
        __syncthreads();
        if (elem) xl = face(W, za - 1, p);
        if (ADJ && elem) xvl = face(V, za - 1, pv);
        __syncthreads();  // plane za - 1 is read before plane za + 1 takes its place
        for (int k = za - 1; k < zb; ++k) {
            if (k + 2 <= zb) fetch(k + 2);
            const bool out = node && k >= za;
            EpiIn1<double> e;
            if (!ADJ && out) epi1_load<double, M>(a, (long long)k * sz + gidx, e);
            double q = 0.0;
            if (elem) {
                const int xu = face(W, k + 1, p + 4);
                const int xvu = ADJ ? face(V, k + 1, pv + 4) : 0;
                double kap = 1.0;
                if (KAPPA) kap = a.kappa[JFNK_IDX(k * n * n + eidx, (long long)n * n * n)];
                const int xm = max(xl, xu), xv = max(xvl, xvu);
                const bool kap_ok = !KAPPA || fx_scale_ok(kap);
                const bool fits = (ADJ ? xm < kFxMaxExp && fx_exp_ok(xv) : fx_exp_ok(xm)) && kap_ok;
                fx_t r[8];
                int Xr = kFxTiny;
                if (fits) {
                    const FxScale sc = KAPPA ? fx_scale_kappa(sc0, kap) : sc0;
                    if (ADJ)
                        fx_vjp3(p, xm, pv, xv, sc, r, Xr);
                    else
                        fx_nd3(p, xm, sc, r, Xr);
                } else {
#pragma unroll
                    for (int c = 0; c < 8; ++c) r[c] = 0;
                    // (a zero element has none, but kappa may be NaN or Inf)
                    if ((ADJ ? xv != 0 || xm == kFxBad : xm != 0) || !kap_ok) {
                        double rs[8];
                        if (ADJ)
                            vjp3_fp64<KAPPA>(a, gx, gy, k, kap, rs);
                        else
                            nd3_fp64<KAPPA, M != Mode::F>(a, eps, gx, gy, k, kap, rs);
#pragma unroll
                        for (int c = 0; c < 8; ++c) r[c] = __double_as_longlong(rs[c]);
                        Xr = kFxFp64;
                    }
                }
                // the lower face's node sums of this layer and the one below
                double d[4];
                if (Xr != kFxFp64 && Xc != kFxFp64) {
                    const int X = max(Xr, Xc) + 1;  // (one bit of room for the sum)
#pragma unroll
                    for (int c = 0; c < 4; ++c) d[c] = fx_to_double(fx_sar(carry[c], X - Xc) + fx_sar(r[c], X - Xr), X);
                } else {
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        d[c] = (Xc == kFxFp64 ? __longlong_as_double(carry[c]) : fx_to_double(carry[c], Xc)) +
                               (Xr == kFxFp64 ? __longlong_as_double(r[c]) : fx_to_double(r[c], Xr));
                }
                double* Ck = C + (k & 1) * 3 * ne + tid;
                q = d[0];          // node (ex, ey)
                Ck[0] = d[1];      // (ex + 1, ey)
                Ck[ne] = d[2];     // (ex, ey + 1)
                Ck[2 * ne] = d[3];  // (ex + 1, ey + 1)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    carry[c] = r[4 + c];
                    p[c] = p[4 + c];
                    if (ADJ) pv[c] = pv[4 + c];
                }
                Xc = Xr;
                xl = xu;
                xvl = xvu;
            }
            if (k + 2 <= zb) store(k + 2);
            __syncthreads();
            if (out) {
                const double* Ck = C + (k & 1) * 3 * ne + tid;
                const double val = (q + Ck[-1]) + (Ck[ne - t.ex] + Ck[2 * ne - t.ex - 1]);
                if (ADJ)
                    epilogue_adj<double, M>(a, (long long)k * sz + gidx, true, val, ck, red);
                else
                    epilogue_pf<double, M>(a, (long long)k * sz + gidx, true, val, inv_eps, ck, e, red);
            }
        }
    }
    stencil_reduce(a, red, red_sm);
}

// Tiling for n elements per direction.  A CTA's time is its layers (planes,
// one more per run, about one of start-up) times a layer's time, which is a
// latency floor plus the element warps that share the SM.
FxTiling fx3d_tiling(const Grid& g) {
    FxTiling best = {};
    if (g.d != 3 || g.beam || g.n < 2 || g.n > 1024) return best;
    const int m = g.n - 1;  // interior nodes per direction
    double best_cost = 1e300;
    for (int tx = 1; tx <= m; ++tx) {
        const int ex = (m + tx - 1) / tx + 1;
        if (ex > 256) continue;
        if (ex < 6 && tx > 1) break;
        for (int cap : {kFxThreads, kFxThreads / 2, kFxThreads / 4, kFxThreads / 8}) {
            int ey = std::min(m + 1, cap / (ex + 1) - 1);  // (ex + 1)(ey + 1) nodes staged
            if (ey < 2) continue;
            const int ty = (m + ey - 2) / (ey - 1);
            ey = (m + ty - 1) / ty + 1;
            FxTiling t = {ex, ey, (m + ex - 2) / (ex - 1), ty, 0, 0, 0};
            t.steps = t.tx * t.ty * m;
            t.threads = (((ex + 1) * (ey + 1) + 31) / 32) * 32;
            const int per_sm = std::max(1, kFxBlocks * kFxThreads / t.threads);
            t.ctas = std::min({t.steps, kNumSMs * per_sm, 2 * kMaxRedBlocks});
            const int planes = (t.steps + t.ctas - 1) / t.ctas;
            const int resident = std::min(per_sm, (t.ctas + kNumSMs - 1) / kNumSMs);
            const double runs = t.tx * t.ty >= t.ctas || t.ctas % (t.tx * t.ty) == 0 ? 1.0 : 1.8;
            const double cost = (planes + 1.7 * runs) * (0.6 + 0.15 * resident * ((ex * ey + 31) / 32));
            if (cost < best_cost) {
                best_cost = cost;
                best = t;
            }
        }
    }
    return best;
}

static bool overlap(const void* p, const void* q, size_t bytes) {
    const char *x = (const char*)p, *y = (const char*)q;
    return p && q && x < y + bytes && y < x + bytes;
}

template <typename T>
bool fx_outputs_alias(const StencilArgs<T>& a, Mode mode) {
    const size_t bytes = sizeof(T) * (size_t)a.g.size;
    const void* in[2] = {a.u, mode == Mode::F ? nullptr : a.v};
    const void* out[3] = {a.out, nullptr, nullptr};
    if (mode == Mode::CHEB || mode == Mode::CHEBLAST) {
        out[0] = a.r;
        out[1] = a.s;
        out[2] = a.dnew;
    } else if (mode == Mode::F || mode == Mode::CHEB0) {
        out[1] = a.out2;
    }
    for (const void* i : in)
        for (const void* o : out)
            if (overlap(i, o, bytes)) return true;
    return false;
}
template bool fx_outputs_alias<double>(const StencilArgs<double>&, Mode);
template bool fx_outputs_alias<float>(const StencilArgs<float>&, Mode);

bool fx3d_use(const StencilArgs<double>& a, Mode mode, bool adj) {
    return a.fx.ctas > 0 && fx_scale_ok(a.node_scale) && !(adj && (a.dkout || mode == Mode::F)) &&
           !fx_outputs_alias(a, mode);
}

template <Prob P, Mode M, bool ADJ>
static jfnk_status launch_fx3d_pm(const StencilArgs<double>& a, cudaStream_t st) {
    const FxTiling& t = a.fx;
    const size_t smem = sizeof(double) * ((ADJ ? 4 : 2) * (size_t)(t.ex + 1) * (t.ey + 1) + 6 * (size_t)t.ex * t.ey);
    fx3d_kernel<P, M, ADJ><<<t.ctas, t.threads, smem, st>>>(a);
    JFNK_LAUNCH_CHECK();
    return JFNK_OK;
}

template <Prob P, bool ADJ>
static jfnk_status launch_fx3d_p(Mode mode, const StencilArgs<double>& a, cudaStream_t st) {
    switch (mode) {
        case Mode::F:
            if constexpr (!ADJ) return launch_fx3d_pm<P, Mode::F, false>(a, st);
            break;
        case Mode::JV: return launch_fx3d_pm<P, Mode::JV, ADJ>(a, st);
        case Mode::BMJ: return launch_fx3d_pm<P, Mode::BMJ, ADJ>(a, st);
        case Mode::CHEB0: return launch_fx3d_pm<P, Mode::CHEB0, ADJ>(a, st);
        case Mode::CHEB: return launch_fx3d_pm<P, Mode::CHEB, ADJ>(a, st);
        case Mode::CHEBLAST: return launch_fx3d_pm<P, Mode::CHEBLAST, ADJ>(a, st);
    }
    set_error("unknown stencil mode");
    return JFNK_ERR_INVALID_ARG;
}

jfnk_status launch_fx3d(Prob prob, Mode mode, bool adj, const StencilArgs<double>& a, cudaStream_t st) {
    if (prob == Prob::ND3)
        return adj ? launch_fx3d_p<Prob::ND3, true>(mode, a, st) : launch_fx3d_p<Prob::ND3, false>(mode, a, st);
    if (prob == Prob::NDK3)
        return adj ? launch_fx3d_p<Prob::NDK3, true>(mode, a, st) : launch_fx3d_p<Prob::NDK3, false>(mode, a, st);
    set_error("the fixed-point kernels evaluate the 3D diffusion problems only");
    return JFNK_ERR_INVALID_ARG;
}

}  // namespace jfnk
