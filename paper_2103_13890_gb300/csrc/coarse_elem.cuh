// Element evaluation of the coarse solvers: the contributions of one element
// from a full-grid vector in (shared) memory.  In FP64 the scalar problems'
// elements run in 64-bit fixed point (fx64.cuh), as on the finer levels: a
// coarse solver runs on a few SMs, whose FP64 pipes would otherwise bound it.
#pragma once
#include "element.cuh"
#include "fx64.cuh"
#include "fx_beam.cuh"
#include "stencil.cuh"

namespace jfnk {

// element contributions per element: 2^d (scalar) or 24 (beam)
__host__ __device__ inline int coarse_npe(const Grid& g) { return g.beam ? 24 : (g.d == 3 ? 8 : 4); }

__device__ __forceinline__ bool coarse_inner(const Grid& g, long long i) { return grid_unknown(g, i); }

// What the fixed-point elements need besides their corners.
template <typename T, Prob P>
struct CoarseElem {
    __device__ explicit CoarseElem(T) {}
};
template <>
struct CoarseElem<double, Prob::BRATU2> {
    bool ok;
    FxBratu b;
    __device__ explicit CoarseElem(double lh) : ok(fx_bratu_ok(lh)), b(fx_bratu(ok ? lh : 0.0)) {}
};
template <>
struct CoarseElem<double, Prob::MINSURF2> {
    bool ok;
    FxMinsurf m;
    __device__ explicit CoarseElem(double lh) : ok(fx_scale_ok(lh)), m(fx_minsurf(ok ? lh : 1.0)) {}
};
template <>
struct CoarseElem<double, Prob::ND3> {
    FxScale s;
    __device__ explicit CoarseElem(double) : s(fx_scale(1.0)) {}
};
template <>
struct CoarseElem<double, Prob::NDK3> {
    FxScale s;
    __device__ explicit CoarseElem(double) : s(fx_scale(1.0)) {}
};

template <>
struct CoarseElem<double, Prob::BEAM3> {
    bool ok;
    FxBeam b;
    __device__ explicit CoarseElem(double inv_h) : ok(fx_scale_ok(inv_h)), b(fx_beam(ok ? inv_h : 1.0)) {}
};

// (out of line: it takes more registers than a coarse solver's thread has)
static __device__ __noinline__ bool coarse_beam_fx(const double* u, const FxBeam& b, double* r) {
    double ue[24], q[24];
    for (int k = 0; k < 24; ++k) ue[k] = u[k];
    if (!fx_neohooke(ue, b, q)) return false;
    for (int k = 0; k < 24; ++k) r[k] = q[k];
    return true;
}

template <typename T, Prob P>
__device__ __forceinline__ void coarse_element_plain(const T* ue, T kap, T lh, T* r) {
    if (P == Prob::MINSURF2)
        elem_minsurf2<T>(ue, lh, r);
    else if (P == Prob::BRATU2)
        elem_bratu2<T>(ue, lh, r);
    else if (P == Prob::NDK3)
        elem_nd3<T, true>(ue, kap, r);
    else
        elem_nd3<T, false>(ue, T(1), r);
}
// out of line: elements outside the fixed-point range
template <Prob P>
__device__ __noinline__ void coarse_element_fp64(const Grid& g, const double* b, double kap, double lh, double* C,
                                                 int cs) {
    constexpr int K = is_2d(P) ? 4 : 8;
    double ue[K], r[K];
    for (int c = 0; c < K; ++c) ue[c] = b[(c & 1) + ((c >> 1) & 1) * g.sy + (c >> 2) * g.sz];
    coarse_element_plain<double, P>(ue, kap, lh, r);
    for (int c = 0; c < K; ++c) C[c * cs] = r[c];
}

// contributions of an element into C[k * cs], k < npe; b: the vector's entry at
// the element's first node (of its first component)
template <typename T, Prob P>
__device__ __forceinline__ void coarse_element_at(const Grid& g, const T* b, T kap, T lh, const CoarseElem<T, P>& ce,
                                                  T* C, int cs) {
    if constexpr (P == Prob::BEAM3) {
        T ue[24], r[24];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const int node = ((c >> 2) * g.ny + ((c >> 1) & 1)) * g.nx + (c & 1);
#pragma unroll
            for (int i = 0; i < 3; ++i) ue[3 * c + i] = b[node * 3 + i];
        }
        bool done = false;
        if constexpr (sizeof(T) == 8) done = ce.ok && coarse_beam_fx(ue, ce.b, r);
        if (!done) elem_neohooke<T>(ue, lh, r);
#pragma unroll
        for (int k = 0; k < 24; ++k) C[k * cs] = r[k];
    } else {
        constexpr int K = is_2d(P) ? 4 : 8;
        const int sy = (int)g.sy, sz = (int)g.sz;
        T ue[K];
#pragma unroll
        for (int c = 0; c < K; ++c) ue[c] = b[(c & 1) + ((c >> 1) & 1) * sy + (c >> 2) * sz];
        if constexpr (sizeof(T) == 8) {
            fx_t p[K], q[K];
            int xm = 0, X = 0;
#pragma unroll
            for (int c = 0; c < K; ++c) {
                p[c] = fx_pack(ue[c]);
                xm = max(xm, fx_exp(p[c]));
            }
            bool done = false;
            if constexpr (P == Prob::BRATU2) {
                const int xe = xm == 0 ? kFxMinExp : xm;
                done = ce.ok && fx_bratu_exp_ok(xe);
                if (done) fx_bratu2(p, xe, ce.b, q, X);
            } else {
                if (xm == 0 && (P != Prob::NDK3 || fx_scale_ok(kap))) {  // contributes zero (kappa is finite)
#pragma unroll
                    for (int c = 0; c < K; ++c) C[c * cs] = T(0);
                    return;
                }
                if constexpr (P == Prob::MINSURF2) {
                    done = ce.ok && fx_exp_ok(xm) && fx_minsurf2(p, xm, ce.m, q, X);
                } else {
                    done = fx_exp_ok(xm) && (P != Prob::NDK3 || fx_scale_ok(kap));
                    if (done) fx_nd3(p, xm, P == Prob::NDK3 ? fx_scale_kappa(ce.s, kap) : ce.s, q, X);
                }
            }
            if (done) {
#pragma unroll
                for (int c = 0; c < K; ++c) C[c * cs] = fx_to_double(q[c], X);
            } else {
                coarse_element_fp64<P>(g, b, kap, lh, C, cs);
            }
        } else {
            T r[K];
            coarse_element_plain<T, P>(ue, kap, lh, r);
#pragma unroll
            for (int c = 0; c < K; ++c) C[c * cs] = r[c];
        }
    }
}

// contributions of element (x, y, z) for the vector w into C[npe]
template <typename T, Prob P>
__device__ __forceinline__ void coarse_element(const Grid& g, const T* w, int x, int y, int z, T kap, T lh,
                                               const CoarseElem<T, P>& ce, T* C) {
    const long long b = P == Prob::BEAM3 ? 3LL * ((z * g.ny + y) * g.nx + x) : z * g.sz + y * g.sy + x;
    coarse_element_at<T, P>(g, w + b, kap, lh, ce, C, 1);
}

}  // namespace jfnk
