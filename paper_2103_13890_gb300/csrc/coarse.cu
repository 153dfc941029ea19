// Coarse-level solve of Algorithm 1 (l = 0): a matrix-free Krylov method in
// place of a direct solver (Sec. 2, "The coarse level solver").  The default
// settings use unrestarted GMRES with x0 = 0; it stops when the Givens
// residual estimate is <= tol ||r0|| (relative reading) or <= tol (absolute),
// or after maxit iterations (Sec. 3: maxit = number of coarse unknowns).
//
// The coarse grid is tiny (<= JFNK_COARSE_MAX_NODES nodes), so the whole solve
// runs in ONE CTA, without kernel launches or host round trips, and an iteration
// is a chain of latencies: barriers, shared-memory reads and dependent FP64
// operations (64 clocks each for one thread).  Hence
//   - the basis holds the unknowns only, and its vectors have unit norm, so
//     that the FD step is the same for all of them;
//   - 8 lanes form a dot product (32 on the larger coarse grids), so that one
//     round of the warps covers a Gram-Schmidt pass;
//   - the Givens rotations of column j, serial FP64 arithmetic, run in a warp of
//     their own while the other warps form the products of iteration j + 1.  The
//     solve stops one (discarded, but counted) iteration after the column that
//     meets the tolerance;
//   - seven barriers an iteration, six of them among the computing warps only.
// Measured (default tolerance; before: a block-wide norm per basis vector, warp-wide
// dot products and the rotations by one thread between the barriers): 5^3 nodes 105
// -> 34 us in FP32 and 171 -> 73 us in FP64, 9^2 nodes 299 -> 72 and 437 -> 143 us,
// 10^3 nodes 670 -> 191 and 1798 -> 780 us.
#include "coarse.cuh"
#include "coarse_elem.cuh"
#include "element.cuh"
#include "reduce.cuh"
#include "stencil.cuh"

namespace jfnk {

// Threads of the one-CTA coarse solvers: the computing warps, one thread per
// node, 256 (32 dot products of 8 lanes at once) to 480, and the warp of the
// Givens rotations.
constexpr int kCoarseMinThreads = 256, kCoarseMaxThreads = 480, kCoarseGivens = 32;
static int coarse_threads(const Grid& g) {
    const long long t = ((g.size + 31) / 32) * 32;
    return (int)(t < kCoarseMinThreads ? kCoarseMinThreads : (t > kCoarseMaxThreads ? kCoarseMaxThreads : t)) +
           kCoarseGivens;
}

// Barrier of the nc computing threads.
__device__ __forceinline__ void coarse_sync(int nc) { asm volatile("bar.sync 1, %0;" ::"r"(nc) : "memory"); }

// Element contributions of the coarse grid, C[c * ne + e]: of A(w), or (ADJ) of
// J(x)^T w.  eoff[e]: where the element's first node is
// in the vectors.
template <typename T, Prob P, bool ADJ>
__device__ __forceinline__ void coarse_elements(const Grid& g, const T* x, const T* w, const unsigned short* eoff, T* C,
                                                int ne, const T* kappa, T lh, const CoarseElem<T, P>& ce, int nc) {
    for (int e = threadIdx.x; e < ne; e += nc) {
        const T kap = P == Prob::NDK3 ? kappa[e] : T(1);
        if constexpr (ADJ) {
            const int sy = (int)g.sy, sz = (int)g.sz;
            T ue[8], ve[8], r[8], dk;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const int i = eoff[e] + (c & 1) + ((c >> 1) & 1) * sy + (c >> 2) * sz;
                ue[c] = x[i];
                ve[c] = w[i];
            }
            elem_vjp3<T>(ue, ve, kap, r, dk);
#pragma unroll
            for (int c = 0; c < 8; ++c) C[c * ne + e] = r[c];
        } else {
            coarse_element_at<T, P>(g, w + eoff[e], kap, lh, ce, C + e, ne);
        }
    }
}

// Sum of the contributions to unknown i (eref: the element whose last corner it
// is).  A scalar grid's unknown has all its elements; the beam's faces do not.
template <typename T, Prob P>
__device__ __forceinline__ T coarse_gather(const Grid& g, const T* C, int ne, int i, int eref) {
    const int n = g.n;
    T acc = T(0);
    if constexpr (P == Prob::BEAM3) {
        const int k = i % 3, node = i / 3, ex = 10 * n;
        const int X = node % g.nx, Y = (node / g.nx) % g.ny, Z = node / (g.nx * g.ny);
        for (int c = 0; c < 8; ++c) {
            const int xe = X - (c & 1), ye = Y - ((c >> 1) & 1), ze = Z - (c >> 2);
            if (xe < 0 || xe >= ex || ye < 0 || ye >= n || ze < 0 || ze >= n) continue;
            acc += C[(3 * c + k) * ne + (ze * n + ye) * ex + xe];
        }
    } else if constexpr (is_2d(P)) {
#pragma unroll
        for (int c = 0; c < 4; ++c) acc += C[(3 - c) * ne + eref + (c & 1) + (c >> 1) * n];
    } else {
#pragma unroll
        for (int c = 0; c < 8; ++c) acc += C[(7 - c) * ne + eref + (c & 1) + ((c >> 1) & 1) * n + (c >> 2) * n * n];
    }
    return acc;
}

// The work of the Givens warp.  One column: the raw entries h1 + h2 (two
// Gram-Schmidt passes) and the squared norm hn2 of what remains; applies the
// earlier rotations, forms the new one and the residual estimate.  Returns
// whether the iteration stops with this column.
struct CoarseGivens {
    double *H, *cs, *sn, *gv, *dinv, *work;  // H: column-major, m + 1 rows
    int m;
    double target;
};
template <typename T>
__device__ bool coarse_givens(const CoarseGivens& s, int j, const T* h1, const T* h2, double hn2) {
    const int lane = threadIdx.x & 31;
    double* const Hj = s.H + (size_t)j * (s.m + 1);
    // r_0 = x_0, r_(i+1) = c_i x_(i+1) - s_i r_i; the rotated entries are c_i r_i + s_i x_(i+1)
    for (int i = lane; i <= j; i += 32) {
        const double x = (double)h1[i] + (double)h2[i];
        Hj[i] = x;
        s.work[i] = i > 0 ? s.cs[i - 1] * x : x;
    }
    __syncwarp();
    double r = s.work[0];
    if (lane == 0 && j > 0) {
        double p = s.work[1], q = s.sn[0];  // (loaded an entry ahead of the chain)
        for (int i = 0; i < j; ++i) {
            const int i1 = i + 1 < j ? i + 1 : i;
            const double p1 = s.work[i1 + 1], q1 = s.sn[i1];
            s.work[i] = r;
            r = fma(-q, r, p);
            p = p1;
            q = q1;
        }
    }
    __syncwarp();
    r = __shfl_sync(0xffffffffu, r, 0);
    for (int i0 = 0; i0 < j; i0 += 32) {
        const int i = i0 + lane;
        double t = 0.0;
        if (i < j) t = fma(s.cs[i], s.work[i], s.sn[i] * Hj[i + 1]);
        __syncwarp();
        if (i < j) Hj[i] = t;  // (entry i0 + 32 is still the raw one the next round reads)
    }
    // 1 / hypot(r, hn), and in lane 1 1 / hn
    const double q2 = lane == 1 ? hn2 : fma(r, r, hn2);
    double ri, hn;
    if (__all_sync(0xffffffffu, q2 >= 1e-280 && q2 <= 1e280)) {
        const double qi = rsqrt_newton(q2);
        ri = __shfl_sync(0xffffffffu, qi, 0);
        const double hi = __shfl_sync(0xffffffffu, qi, 1), h0 = hn2 * hi;
        hn = fma(fma(-h0, h0, hn2), 0.5 * hi, h0);
    } else {
        hn = sqrt(hn2);
        ri = 1.0 / hypot(r, hn);
    }
    double c = 1.0, sg = 0.0, d = r, di = ri;
    if (hn != 0.0) {
        c = r * ri;
        sg = hn * ri;
        d = fma(c, r, sg * hn);
    } else {
        di = 1.0 / r;
    }
    const double g = s.gv[j], gn = -sg * g;
    __syncwarp();
    if (lane == 0) {
        Hj[j] = d;
        s.cs[j] = c;
        s.sn[j] = sg;
        s.dinv[j] = di;
        s.gv[j + 1] = gn;
        s.gv[j] = c * g;
    }
    __syncwarp();
    const double res = fabs(gn);
    return res <= s.target || !(hn > 0.0) || !isfinite(res);
}

// vsm: the Krylov basis V and the Hessenberg matrix H live in shared memory
// (after the work arrays) instead of the global scratch a.V / a.H
template <typename T, Prob P, bool ADJ>
__device__ void coarse_gmres_body(const CoarseArgs<T>& a, unsigned char* smem_raw, bool vsm) {
    const Grid g = a.g;
    const int N = (int)g.size, U = (int)g.interior();
    const int ne = (int)g.elements();
    const int npe = coarse_npe(g);
    const int m = a.maxit;
    CoarseGivens gs;
    gs.m = m;
    gs.cs = reinterpret_cast<double*>(smem_raw);  // [m]
    gs.sn = gs.cs + m;                            // [m]
    gs.dinv = gs.sn + m;                          // [m]
    gs.gv = gs.dinv + m;                          // [m + 1]
    gs.work = gs.gv + (m + 1);                    // [m + 1]
    double* const red = gs.work + (m + 1);        // [32]
    T* const part = reinterpret_cast<T*>(red);    // [2][16] squared norms of the warps by column parity
    gs.H = a.H;
    double* end = red + 32;
    if (vsm) {
        gs.H = end;
        end += (size_t)(m + 1) * m;
    }
    T* const x = reinterpret_cast<T*>(end);  // [N] x_0
    T* const xw = x + N;                     // [N] x_0 + eps v (ADJ: v)
    T* const Ax = xw + N;                    // [U] A(x_0)
    T* const wv = Ax + U;                    // [U] work vector
    T* const hp = wv + U;                    // [2][2][m + 1] dot products by column parity and pass
    T* const C = hp + 4 * (m + 1);           // [npe * ne]
    T* const V = vsm ? C + npe * ne : a.V;   // [m + 1][U]
    unsigned short* const idx = reinterpret_cast<unsigned short*>(vsm ? V + (size_t)(m + 1) * U : C + npe * ne);
    unsigned short* const eref = idx + U;    // [U]
    unsigned short* const eoff = eref + U;   // [ne]
    __shared__ int s_flag[2];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int nc = blockDim.x - kCoarseGivens, nw = nc >> 5;
    const bool comp = tid < nc;
    constexpr int LU = sizeof(T) == 8 ? 2 : 1;      // lanes of an unknown's update
    const int nwu = min(nw, (U * LU + 31) / 32);    // warps with unknowns
    // squared norm of what remains of column j, by the Givens warp
    auto remains = [&](int j) { return warp_sum(lane < nwu ? (double)part[(j & 1) * 16 + lane] : 0.0); };

    // ||b|| over the unknowns; V_0 = b / ||b||
    double acc = 0.0;
    for (int i = tid; i < N; i += blockDim.x)
        if (coarse_inner(g, i)) acc += (double)a.b[i] * (double)a.b[i];
    __shared__ double s_beta[2], s_eps[2];
    if (tid == 32) {  // the FD step of a unit vector
        const double e = eps_formula(a.eps_mode, a.n_unknowns, *a.xstat, 1.0);
        s_eps[0] = e;
        s_eps[1] = e > 0.0 ? 1.0 / e : 0.0;
    }
    const double bn = block_sum(acc, red);
    if (tid == 0) {
        s_beta[0] = sqrt(bn);
        s_beta[1] = 1.0 / s_beta[0];
    }
    __syncthreads();
    const double beta = s_beta[0];
    const double target = a.tol_abs ? a.tol : a.tol * beta;
    gs.target = target;
    if (!(beta > 0.0) || beta <= target) {
        for (int i = tid; i < N; i += blockDim.x) a.s[i] = T(0);
        return;
    }
    if (wid == nw) {  // the unknowns in order
        int base = 0;
        for (int i0 = 0; i0 < N; i0 += 32) {
            const int i = i0 + lane;
            const bool in = i < N && coarse_inner(g, i);
            const unsigned int mask = __ballot_sync(0xffffffffu, in);
            if (in) {
                const int u = base + __popc(mask & ((1u << lane) - 1));
                const int X = i % g.nx, Y = (i / g.nx) % g.ny, Z = i / (g.nx * g.ny);
                idx[u] = (unsigned short)i;
                eref[u] = P == Prob::BEAM3 ? 0 : (unsigned short)(((g.d == 3 ? Z - 1 : 0) * g.n + Y - 1) * g.n + X - 1);
            }
            base += __popc(mask);
        }
        for (int j = lane; j <= m; j += 32) gs.gv[j] = j == 0 ? beta : 0.0;
    } else {
        const int ex = P == Prob::BEAM3 ? 10 * g.n : g.n;
        for (int e = tid; e < ne; e += nc) {
            const int X = e % ex, Y = (e / ex) % g.n, Z = e / (ex * g.n);
            eoff[e] = (unsigned short)(P == Prob::BEAM3 ? 3 * ((Z * g.ny + Y) * g.nx + X) : Z * (int)g.sz + Y * (int)g.sy + X);
        }
        for (int i = tid; i < N; i += nc) {
            x[i] = a.x[i];
            xw[i] = ADJ ? T(0) : a.x[i];
        }
    }
    __syncthreads();
    const T eps = (T)s_eps[0], inv_eps = (T)s_eps[1];
    if (comp) {
        const double bi = s_beta[1];
        for (int u = tid; u < U; u += nc) {
            const int i = idx[u];
            double q = (double)a.b[i] * bi;
            if (sizeof(T) == 8) q = fma(fma(-q, beta, (double)a.b[i]), bi, q);  // (the quotient's rounding alone)
            const T v = (T)q;
            V[u] = v;
            if (!ADJ) Ax[u] = a.Ax[i];
            xw[i] = ADJ ? v : x[i] + eps * v;
        }
    }
    __syncthreads();
    const CoarseElem<T, P> ce(a.lh);
    const int lg = U <= 128 ? 3 : 5, dl = 1 << lg;  // lanes of a dot product
    int k = 0, formed = 0;  // columns, products
    // (dots and updates in the basis precision T: in an FP32 preconditioner the
    // single CTA would otherwise spend its iterations on this SM's FP64 pipe,
    // 1/74 of the FP32 rate; the Hessenberg entries are kept in FP64)
    for (int j = 0; j < m; ++j) {
        T* const hj = hp + (j & 1) * 2 * (m + 1);
        if (comp) {
            coarse_elements<T, P, ADJ>(g, x, xw, eoff, C, ne, a.kappa, a.lh, ce, nc);
            coarse_sync(nc);
            for (int u = tid; u < U; u += nc) {
                T w = coarse_gather<T, P>(g, C, ne, idx[u], eref[u]);
                if (P != Prob::BEAM3) w *= a.node_scale;
                wv[u] = ADJ ? w : (w - Ax[u]) * inv_eps;
            }
            coarse_sync(nc);
            // classical Gram-Schmidt, twice
            T n2 = T(0);
            for (int pass = 0; pass < 2; ++pass) {
                T* const h = hj + pass * (m + 1);
                for (int q0 = wid * (32 >> lg); q0 <= j; q0 += nw * (32 >> lg)) {
                    const int q = q0 + (lane >> lg);
                    T d = T(0);
                    if (q <= j) {
                        const T* const vq = V + q * U;
                        for (int u = lane & (dl - 1); u < U; u += dl) d += wv[u] * vq[u];
                    }
                    for (int o = dl >> 1; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
                    if (q <= j && (lane & (dl - 1)) == 0) h[q] = d;
                }
                coarse_sync(nc);
                for (int u0 = 0; u0 < U; u0 += nc / LU) {
                    const int u = u0 + tid / LU;
                    if (u0 + wid * (32 / LU) >= U) continue;  // (whole warps)
                    const T* const vu = V + (u < U ? u : 0);
                    T s0 = T(0), s1 = T(0);
                    int q = tid % LU;
                    for (; q + LU <= j; q += 2 * LU) {
                        s0 += h[q] * vu[q * U];
                        s1 += h[q + LU] * vu[(q + LU) * U];
                    }
                    if (q <= j) s0 += h[q] * vu[q * U];
                    s0 += s1;
                    if (LU == 2) s0 += __shfl_xor_sync(0xffffffffu, s0, 1);
                    if (u < U && tid % LU == 0) {
                        const T w = wv[u] - s0;
                        wv[u] = w;
                        if (pass == 1) n2 += w * w;
                    }
                }
                if (pass == 0) coarse_sync(nc);
            }
            // the squared norm of what remains
            T* const pj = part + (j & 1) * 16;
            if (wid < nwu) {
                n2 = warp_sum(n2);
                if (lane == 0) pj[wid] = n2;
            }
            coarse_sync(nc);
            if (j + 1 < m && tid < U) {
                const T hinv = coarse_rsqrt(pj, nwu);
                T* const vn = V + (j + 1) * U;
                for (int u = tid; u < U; u += nc) {
                    const int i = idx[u];
                    const T v = wv[u] * hinv;
                    vn[u] = v;
                    xw[i] = ADJ ? v : x[i] + eps * v;
                }
            }
        } else if (j > 0) {
            const int pj = (j - 1) & 1;
            const T* const h = hp + pj * 2 * (m + 1);
            const bool stop = coarse_givens<T>(gs, j - 1, h, h + m + 1, remains(j - 1));
            if (lane == 0) s_flag[pj] = stop;
        }
        __syncthreads();
        k = formed = j + 1;
        if (j > 0 && s_flag[(j - 1) & 1]) {
            k = j;
            break;
        }
    }
    // the last column, if the loop ran to its end; back-substitution,
    // y into hp
    if (!comp) {
        if (k == m) {
            const int pj = (m - 1) & 1;
            const T* const h = hp + pj * 2 * (m + 1);
            coarse_givens<T>(gs, m - 1, h, h + m + 1, remains(m - 1));
        }
        for (int i = k - 1; i >= 0; --i) {
            const double* const Hi = gs.H + (size_t)i * (m + 1);
            const double y = gs.gv[i] * gs.dinv[i];
            __syncwarp();
            if (lane == 0) gs.gv[i] = y;
            for (int q = lane; q < i; q += 32) gs.gv[q] = fma(-Hi[q], y, gs.gv[q]);
            __syncwarp();
        }
        for (int q = lane; q < k; q += 32) hp[q] = (T)gs.gv[q];
        if (lane == 0 && a.iters) *a.iters += formed;
    } else {
        for (int i = tid; i < N; i += nc)
            if (!coarse_inner(g, i)) a.s[i] = T(0);
    }
    __syncthreads();
    for (int u = tid; u < U; u += blockDim.x) {
        T s0 = T(0), s1 = T(0);
        int q = 0;
        for (; q + 1 < k; q += 2) {
            s0 += hp[q] * V[q * U + u];
            s1 += hp[q + 1] * V[(q + 1) * U + u];
        }
        if (q < k) s0 += hp[q] * V[q * U + u];
        a.s[idx[u]] = s0 + s1;
    }
}

template <typename T, Prob P, bool ADJ>
__global__ void __launch_bounds__(kCoarseMaxThreads + kCoarseGivens) coarse_gmres_kernel(CoarseArgs<T> a, int vsm) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    coarse_gmres_body<T, P, ADJ>(a, smem_raw, vsm != 0);
}

// one CTA per instance of a batch (all instances share the coarse grid size)
template <typename T, Prob P, bool ADJ>
__global__ void __launch_bounds__(kCoarseMaxThreads + kCoarseGivens) coarse_gmres_batched_kernel(const CoarseArgs<T>* args, int vsm) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const CoarseArgs<T> a = args[blockIdx.x];
    coarse_gmres_body<T, P, ADJ>(a, smem_raw, vsm != 0);
}

// Shared memory of the GMRES kernel: work arrays, plus V and H when vsm.
template <typename T>
size_t coarse_smem_bytes(const Grid& g, int maxit, bool vsm) {
    const size_t ne = (size_t)g.elements(), u = (size_t)g.interior(), m = (size_t)maxit;
    size_t b = sizeof(double) * (5 * m + 2 + 32);
    b += sizeof(T) * (2 * (size_t)g.size + 2 * u + 4 * (m + 1) + ne * coarse_npe(g));
    b += sizeof(unsigned short) * (2 * u + ne);
    if (vsm) b += sizeof(double) * (m + 1) * m + sizeof(T) * (m + 1) * u;
    return b;
}

// V and H go to shared memory when everything fits in kCoarseVsmBytes (the
// basis is then read at shared-memory rather than L2 latency in the
// orthogonalisation, the critical path of this one-CTA solver)
constexpr size_t kCoarseVsmBytes = 160 * 1024;
template <typename T>
static bool coarse_vsm(const Grid& g, int maxit) {
    return coarse_smem_bytes<T>(g, maxit, true) <= kCoarseVsmBytes;
}

template <typename T>
jfnk_status launch_coarse(Prob prob, const CoarseArgs<T>& a, cudaStream_t st) {
    if (a.g.size > JFNK_COARSE_MAX_NODES || a.maxit > JFNK_COARSE_MAX_IT || a.maxit < 1) {
        set_error("coarse grid too large for the single-CTA solver (%lld nodes, maxit %d)", a.g.size, a.maxit);
        return JFNK_ERR_INVALID_ARG;
    }
    if (a.method == 1) return launch_coarse_cgqn<T>(prob, a, st);
    const bool vsm = coarse_vsm<T>(a.g, a.maxit);
    const size_t smem = coarse_smem_bytes<T>(a.g, a.maxit, vsm);
    if (smem > 200 * 1024) {
        set_error("coarse solver shared memory %zu too large", smem);
        return JFNK_ERR_INVALID_ARG;
    }
    if (a.adjoint && is_2d(prob)) {
        set_error("the adjoint coarse solve is implemented for the 3D diffusion problems");
        return JFNK_ERR_NOT_IMPLEMENTED;
    }
#define JFNK_COARSE_LAUNCH(PP, ADJ)                                                                  \
    do {                                                                                             \
        JFNK_CUDA_TRY(cudaFuncSetAttribute(coarse_gmres_kernel<T, PP, ADJ>,                           \
                                           cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)); \
        coarse_gmres_kernel<T, PP, ADJ><<<1, coarse_threads(a.g), smem, st>>>(a, vsm ? 1 : 0);             \
    } while (0)
    switch (prob) {
        case Prob::BRATU2: JFNK_COARSE_LAUNCH(Prob::BRATU2, false); break;
        case Prob::MINSURF2: JFNK_COARSE_LAUNCH(Prob::MINSURF2, false); break;
        case Prob::BEAM3:
            if (a.adjoint) {
                set_error("no adjoint for the beam");
                return JFNK_ERR_NOT_IMPLEMENTED;
            }
            JFNK_COARSE_LAUNCH(Prob::BEAM3, false);
            break;
        case Prob::ND3:
            if (a.adjoint) JFNK_COARSE_LAUNCH(Prob::ND3, true);
            else JFNK_COARSE_LAUNCH(Prob::ND3, false);
            break;
        case Prob::NDK3:
            if (a.adjoint) JFNK_COARSE_LAUNCH(Prob::NDK3, true);
            else JFNK_COARSE_LAUNCH(Prob::NDK3, false);
            break;
    }
#undef JFNK_COARSE_LAUNCH
    JFNK_LAUNCH_CHECK();
    return JFNK_OK;
}

template jfnk_status launch_coarse<float>(Prob, const CoarseArgs<float>&, cudaStream_t);
template jfnk_status launch_coarse<double>(Prob, const CoarseArgs<double>&, cudaStream_t);
template <typename T>
jfnk_status launch_coarse_batched(const CoarseArgs<T>& a0, const CoarseArgs<T>* dev_args, int count, cudaStream_t st) {
    if (count <= 0) return JFNK_OK;
    if (a0.g.size > JFNK_COARSE_MAX_NODES || a0.maxit > JFNK_COARSE_MAX_IT || a0.maxit < 1 || a0.g.d != 2) {
        set_error("batched coarse solve: 2D coarse grids within the single-CTA limits only");
        return JFNK_ERR_INVALID_ARG;
    }
    const bool vsm = coarse_vsm<T>(a0.g, a0.maxit);
    const size_t smem = coarse_smem_bytes<T>(a0.g, a0.maxit, vsm);
    JFNK_CUDA_TRY(cudaFuncSetAttribute(coarse_gmres_batched_kernel<T, Prob::BRATU2, false>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    coarse_gmres_batched_kernel<T, Prob::BRATU2, false><<<count, coarse_threads(a0.g), smem, st>>>(dev_args,
                                                                                                   vsm ? 1 : 0);
    JFNK_LAUNCH_CHECK();
    return JFNK_OK;
}
template jfnk_status launch_coarse_batched<float>(const CoarseArgs<float>&, const CoarseArgs<float>*, int, cudaStream_t);
template jfnk_status launch_coarse_batched<double>(const CoarseArgs<double>&, const CoarseArgs<double>*, int, cudaStream_t);

}  // namespace jfnk
