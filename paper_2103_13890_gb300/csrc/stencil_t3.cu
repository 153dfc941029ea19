// FP32 residual of the 3D diffusion problems and its vector-Jacobian product:
// z-marching tiles, two elements a thread in packed FP32 arithmetic, one launch
// per action.
//
// A CTA takes a tile of ex x ey element columns (ey even); thread (tx, ty)
// evaluates the elements of rows 2 ty and 2 ty + 1 as one packed pair
// (pf2.cuh), so that the row between them is summed in registers.  Node planes
// (w = x + eps v; for the product also the direction) are staged in shared
// memory, contributions to the upper face stay in registers for the next layer,
// and what a thread holds for the columns beside it goes through shared memory:
// 4 stores and 4 loads a pair.  One barrier a layer, everything double-buffered.
// Tiles overlap by one element, and the (tile, plane) pairs are dealt to the
// CTAs in equal contiguous runs, as in the FP64 kernel (stencil_fx.cu).
//
// Bound by the FMA pipe and instruction issue (257^3 residual: FMA pipe 54 %,
// issue slots about half, DRAM 16 %).  Against the halo-free pair of kernels with
// its face fixup (stencil_v2.cu) and the element-parallel pair on smaller levels
// (stencil_ep.cu): residual 257^3 215 -> 164 us, 129^3 31 -> 27 us, 33^3 11.2 ->
// 8.2 us; FD action 257^3 240 -> 179 us; vector-Jacobian product 257^3 407 -> 245,
// 129^3 57 -> 37 us.  One CTA of up to 512 threads per SM: 256 x 2 took 183 us for
// the 257^3 residual, 192 x 3 203, 128 x 5 182.
#include <algorithm>

#include "element.cuh"
#include "pf2.cuh"
#include "reduce.cuh"
#include "stencil.cuh"
#include "stencil_body.cuh"
#include "stencil_fx.cuh"
#include "stencil_t3.cuh"

namespace jfnk {

// Smaller levels run in one CTA (n <= 8), in one cluster (n = 16) or, 9 to 15, in the
// element-parallel pair (stencil_ep.cu).  A smoothing step with its norm takes 8.3-8.4
// us here and in a cluster for n = 10 to 20 alike, 10.4 us in the pair; the pair on 9 to
// 15 predates both and is the slower one.
constexpr int kT3MinN = 17;
constexpr int kT3Threads = 512;  // largest CTA (128 registers a thread)

template <Prob P, Mode M, bool ADJ>
__global__ void __launch_bounds__(kT3Threads, 1) t3d_kernel(const StencilArgs<float> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double red_sm[32];
    constexpr bool KAPPA = P == Prob::NDK3;
    const FxTiling& t = a.t3;
    const int n = a.g.n;
    const int sy = (int)a.g.sy, sz = (int)a.g.sz;
    const int npx = t.ex + 1, npy = t.ey + 1, np = npx * npy, eyp = t.ey >> 1;
    float* const W = reinterpret_cast<float*>(smem_raw);  // [2][np]: w (not ADJ: times kNd3FaceCorner)
    float* const V = W + (ADJ ? 2 * np : 0);              // [2][np]: direction (ADJ)
    const int cb = (eyp + 1) * npx;
    float* const CA = V + 2 * np;                         // [2][np]: rows 2 ty, 2 ty + 1 from the left column
    float* const CB = CA + 2 * np;                        // [2][2][cb]: row 2 ty from the pair below, a = 0 / 1
    const int tid = threadIdx.x;
    float eps = 0.f, inv_eps = 0.f;
    if (!ADJ && M != Mode::F) {
        eps = eps_of<float>(a.eps);
        inv_eps = inv_eps_of<float>(a.eps);
    }
    ChebK<float> ck = {0.f, 0.f, 0.f};
    if (M == Mode::CHEB0 || M == Mode::CHEB || M == Mode::CHEBLAST) ck = cheb_of<float>(a.cheb, a.cheb_step);
    const int tx = tid % t.ex, ty = tid / t.ex;
    const bool active = tid < t.ex * eyp;
    const int at = 2 * ty * npx + tx;  // own corner in a plane
    // the plane's last column and row, one extra node for the first npy + ex threads
    const int xx = tid < npy ? t.ex : tid - npy, xy = tid < npy ? tid : t.ey;
    const bool extra = tid < npy + t.ex;
    const float scale = ADJ ? a.node_scale : (float)(a.node_scale * kNd3FaceScale);
    float red = 0.f;

    int step = (int)((long long)t.steps * blockIdx.x / gridDim.x);
    const int last = (int)((long long)t.steps * (blockIdx.x + 1) / gridDim.x);
    while (step < last) {
        const int tile = step / (n - 1);
        const int za = step - tile * (n - 1) + 1;   // first plane of this run
        const int zb = min(n, za + (last - step));  // one past its last
        step += zb - za;
        const int x0 = (tile % t.tx) * (t.ex - 1), y0 = (tile / t.tx) * (t.ey - 1);
        const int X = x0 + tx, Y = y0 + 2 * ty;
        // this thread's nodes of a staged plane: (X, Y), (X, Y + 1) and the extra
        // one; `inside`: in the grid, `dir`: unknowns in x and y
        const int XX = x0 + xx, XY = y0 + xy;
        const bool in0 = active && X <= n && Y <= n, in1 = active && X <= n && Y < n, in2 = extra && XX <= n && XY <= n;
        auto unknown = [&](int x, int y) { return x > 0 && x < n && y > 0 && y < n; };
        const bool dir0 = in0 && unknown(X, Y), dir1 = in1 && unknown(X, Y + 1), dir2 = in2 && unknown(XX, XY);
        const bool rim = x0 == 0 || y0 == 0 || x0 + t.ex >= n || y0 + t.ey >= n;  // (CTA-uniform) some are not
        const int j0 = Y * sy + X, j2 = XY * sy + XX;
        float u0 = 0.f, u1 = 0.f, u2 = 0.f, v0 = 0.f, v1 = 0.f, v2 = 0.f;
        auto fetch = [&](int z) {
            const float* pu = a.u + (long long)z * sz;
            if (in0) u0 = pu[JFNK_IDX(j0, sz)];
            if (in1) u1 = pu[JFNK_IDX(j0 + sy, sz)];
            if (in2) u2 = pu[JFNK_IDX(j2, sz)];
            if (ADJ || M != Mode::F) {
                const float* pv = a.v + (long long)z * sz;
                const bool zin = z > 0 && z < n;
                v0 = dir0 && zin ? pv[JFNK_IDX(j0, sz)] : 0.f;
                v1 = dir1 && zin ? pv[JFNK_IDX(j0 + sy, sz)] : 0.f;
                if (in2) v2 = dir2 && zin ? pv[JFNK_IDX(j2, sz)] : 0.f;
            }
        };
        // (the scaling of the corner values is exact)
        auto wv = [&](float u, float v) {
            if (ADJ) return u;
            const float c = (float)kNd3FaceCorner * u;
            return M != Mode::F ? fmaf((float)kNd3FaceCorner * eps, v, c) : c;
        };
        auto store = [&](int z) {
            float* Wz = W + (z & 1) * np;
            float* Vz = V + (z & 1) * np;
            if (active) {
                Wz[at] = wv(u0, v0);
                Wz[at + npx] = wv(u1, v1);
                if (ADJ) {
                    Vz[at] = v0;
                    Vz[at + npx] = v1;
                }
            }
            if (extra) {
                Wz[xy * npx + xx] = wv(u2, v2);
                if (ADJ) Vz[xy * npx + xx] = v2;
            }
            if (rim || z == 0 || z == n) {  // Dirichlet nodes: every output is zero
                const bool zb0 = z == 0 || z == n;
                auto zero = [&](int j) {
                    if (ADJ)
                        epilogue_adj<float, M>(a, (long long)z * sz + j, false, 0.f, ck, red);
                    else
                        epilogue<float, M>(a, (long long)z * sz + j, false, 0.f, 0.f, ck, red);
                };
                if (in0 && (zb0 || !dir0)) zero(j0);
                if (in1 && (zb0 || !dir1)) zero(j0 + sy);
                if (in2 && (zb0 || !dir2)) zero(j2);
            }
        };
        // packed corners (a, b) of a plane: lo the element of row Y, hi of row Y + 1
        auto face = [&](const float* plane, int z, pf2* q) {
            const float* p = plane + (z & 1) * np + at;
            const float r0 = p[0], r1 = p[npx], r2 = p[2 * npx], s0 = p[1], s1 = p[npx + 1], s2 = p[2 * npx + 1];
            q[0] = pf2_pack(r0, r1);
            q[1] = pf2_pack(s0, s1);
            q[2] = pf2_pack(r1, r2);
            q[3] = pf2_pack(s1, s2);
        };
        const bool outx = active && tx > 0 && X < n;
        const bool ok0 = outx && ty > 0 && Y < n, ok1 = outx && Y + 1 < n;
        pf2 w[8], v[8], carry[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) carry[c] = pf2(0.0);
        fetch(za - 1);
        store(za - 1);
        fetch(za);
        store(za);
        __syncthreads();
        if (active) {
            face(W, za - 1, w);
            if (ADJ) {
                face(V, za - 1, v);
            } else {
                pf2 m[4];
                nd3_face(w, m);
#pragma unroll
                for (int c = 0; c < 4; ++c) w[c] = m[c];  // the lower face as modes
            }
        }
        __syncthreads();  // plane za - 1 is read before plane za + 1 takes its place
        for (int k = za - 1; k < zb; ++k) {
            if (k + 2 <= zb) fetch(k + 2);
            const bool out0 = ok0 && k >= za, out1 = ok1 && k >= za;
            EpiIn1<float> e0, e1;
            if (!ADJ) {
                if (out0) epi1_load<float, M>(a, (long long)k * sz + j0, e0);
                if (out1) epi1_load<float, M>(a, (long long)k * sz + j0 + sy, e1);
            }
            float s0 = 0.f, s1 = 0.f;
            if (active) {
                face(W, k + 1, w + 4);
                pf2 kap = pf2(1.0);
                if (KAPPA) {
                    const int e = (k * n + Y) * n + X;
                    kap = pf2_pack(X < n && Y < n ? a.kappa[JFNK_IDX(e, (long long)n * n * n)] : 0.f,
                                   X < n && Y + 1 < n ? a.kappa[JFNK_IDX(e + n, (long long)n * n * n)] : 0.f);
                }
                pf2 r[4];  // node plane k: this layer and the one below
                if (ADJ) {
                    face(V, k + 1, v + 4);
                    pf2 q[8], dk;
                    elem_vjp3<pf2>(w, v, kap, q, dk);
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        r[c] = carry[c] + q[c];
                        carry[c] = q[4 + c];
                        w[c] = w[4 + c];
                        v[c] = v[4 + c];
                    }
                } else {
                    pf2 up[4], lt[4], ut[4], sum[4];
                    nd3_face(w + 4, up);
                    nd3_faces<pf2, KAPPA>(w, up, kap, lt, ut);
                    sum[0] = carry[0] - lt[0];
#pragma unroll
                    for (int c = 1; c < 4; ++c) sum[c] = carry[c] + lt[c];
                    nd3_face_adj(sum, r);
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        carry[c] = ut[c];
                        w[c] = up[c];
                    }
                }
                float lo[4], hi[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) pf2_unpack(r[c], lo[c], hi[c]);
                s0 = lo[0];
                s1 = lo[2] + hi[0];
                float* A = CA + (k & 1) * np + at + 1;
                A[0] = lo[1];
                A[npx] = lo[3] + hi[1];
                float* B = CB + (k & 1) * 2 * cb + (ty + 1) * npx + tx;
                B[0] = hi[2];
                B[cb + 1] = hi[3];
            }
            if (k + 2 <= zb) store(k + 2);
            __syncthreads();
            const float* A = CA + (k & 1) * np + at;
            const float* B = CB + (k & 1) * 2 * cb + ty * npx + tx;
            const long long i0 = (long long)k * sz + j0;
            if (out0) {
                const float val = ((s0 + A[0]) + (B[0] + B[cb])) * scale;
                if (ADJ)
                    epilogue_adj<float, M>(a, i0, true, val, ck, red);
                else
                    epilogue_pf<float, M>(a, i0, true, val, inv_eps, ck, e0, red);
            }
            if (out1) {
                const float val = (s1 + A[npx]) * scale;
                if (ADJ)
                    epilogue_adj<float, M>(a, i0 + sy, true, val, ck, red);
                else
                    epilogue_pf<float, M>(a, i0 + sy, true, val, inv_eps, ck, e1, red);
            }
        }
    }
    stencil_reduce(a, red, red_sm);
}

// Tiling for n elements per direction: as for the FP64 kernel, a CTA's time is
// its layers (planes, one more per run, about one of start-up) times a layer's,
// a latency floor plus the warps that share the SM.
FxTiling t3d_tiling(const Grid& g) {
    FxTiling best = {};
    if (g.d != 3 || g.beam || g.n < kT3MinN || g.n > 1024) return best;
    const int m = g.n - 1;
    double best_cost = 1e300;
    for (int tx = 1; tx <= m; ++tx) {
        const int ex = (m + tx - 1) / tx + 1;
        if (ex > 128) continue;
        if (ex < 6 && tx > 1) break;
        for (int cap : {kT3Threads, kT3Threads / 2, kT3Threads / 4, kT3Threads / 8}) {
            int ep = std::min((m + 2) / 2, cap / ex);  // element row pairs
            if (ep < 1) continue;
            const int ty = (m + 2 * ep - 2) / (2 * ep - 1);
            ep = ((m + ty - 1) / ty + 2) / 2;
            const int ey = 2 * ep;
            FxTiling t = {ex, ey, (m + ex - 2) / (ex - 1), (m + ey - 2) / (ey - 1), 0, 0, 0};
            t.steps = t.tx * t.ty * m;
            // (a thread stages at most one node of the last column and row)
            t.threads = ((std::max(ex * ep, ex + ey + 1) + 31) / 32) * 32;
            if (t.threads > kT3Threads) continue;
            const int per_sm = std::max(1, kT3Threads / t.threads);
            t.ctas = std::min({t.steps, kNumSMs * per_sm, 2 * kMaxRedBlocks});
            const int planes = (t.steps + t.ctas - 1) / t.ctas;
            const int resident = std::min(per_sm, (t.ctas + kNumSMs - 1) / kNumSMs);
            const double runs = t.tx * t.ty >= t.ctas || t.ctas % (t.tx * t.ty) == 0 ? 1.0 : 1.8;
            const double cost = (planes + 1.7 * runs) * (0.4 + 0.035 * resident * ((ex * ep + 31) / 32));
            if (cost < best_cost) {
                best_cost = cost;
                best = t;
            }
        }
    }
    return best;
}

bool t3d_use(const StencilArgs<float>& a, Mode mode, bool adj) {
    return a.t3.ctas > 0 && !(adj && (a.dkout || mode == Mode::F)) && !fx_outputs_alias(a, mode);
}

template <Prob P, Mode M, bool ADJ>
static jfnk_status launch_t3d_pm(const StencilArgs<float>& a, cudaStream_t st) {
    const FxTiling& t = a.t3;
    const size_t np = (size_t)(t.ex + 1) * (t.ey + 1), cb = (size_t)(t.ey / 2 + 1) * (t.ex + 1);
    const size_t smem = sizeof(float) * ((ADJ ? 6 : 4) * np + 4 * cb + 4);
    t3d_kernel<P, M, ADJ><<<t.ctas, t.threads, smem, st>>>(a);
    JFNK_LAUNCH_CHECK();
    return JFNK_OK;
}

template <Prob P, bool ADJ>
static jfnk_status launch_t3d_p(Mode mode, const StencilArgs<float>& a, cudaStream_t st) {
    switch (mode) {
        case Mode::F:
            if constexpr (!ADJ) return launch_t3d_pm<P, Mode::F, false>(a, st);
            break;
        case Mode::JV: return launch_t3d_pm<P, Mode::JV, ADJ>(a, st);
        case Mode::BMJ: return launch_t3d_pm<P, Mode::BMJ, ADJ>(a, st);
        case Mode::CHEB0: return launch_t3d_pm<P, Mode::CHEB0, ADJ>(a, st);
        case Mode::CHEB: return launch_t3d_pm<P, Mode::CHEB, ADJ>(a, st);
        case Mode::CHEBLAST: return launch_t3d_pm<P, Mode::CHEBLAST, ADJ>(a, st);
    }
    set_error("mode not available for the tiled FP32 kernels");
    return JFNK_ERR_INVALID_ARG;
}

jfnk_status launch_t3d(Prob prob, Mode mode, bool adj, const StencilArgs<float>& a, cudaStream_t st) {
    if (prob == Prob::ND3)
        return adj ? launch_t3d_p<Prob::ND3, true>(mode, a, st) : launch_t3d_p<Prob::ND3, false>(mode, a, st);
    if (prob == Prob::NDK3)
        return adj ? launch_t3d_p<Prob::NDK3, true>(mode, a, st) : launch_t3d_p<Prob::NDK3, false>(mode, a, st);
    set_error("the tiled FP32 kernels evaluate the 3D diffusion problems only");
    return JFNK_ERR_INVALID_ARG;
}

}  // namespace jfnk
