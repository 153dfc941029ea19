// The paper's coarse solver (Sec. 2 "The coarse level solver", Alg. 1, l = 0):
// CG preconditioned by L-BFGS, stopped on negative curvature, and re-run on the
// shifted operator A_s = A - lambda_c+ I (lambda_c+ <= 0) with
// lambda_c+ <- gamma min(lambda_c, lambda_c+) while the Rayleigh quotient
// lambda_c = p.A_s p / p.p of the direction of negative curvature is < 0.
// The secant pairs (s_i, y_i) = (alpha_i p_i, alpha_i A p_i) of the very first
// call are collected; m of the k steps, those of iterations floor(j k / m),
// are kept (uniform sampling) and define the preconditioner for the rest of
// the solve.  Each shifted call restarts CG from the returned s_0.  At most
// 30 shifted calls.
//
// One thread-block cluster runs the whole solve.  Every CTA owns a contiguous
// slice of the unknowns, in its shared memory: the CG vectors and its part of
// the kept pairs.  p is pushed to every CTA's copy of the full vector
// (distributed shared memory); each CTA sums p.p for the FD step and the Rayleigh
// quotient, forms x_0 + eps p, and evaluates the elements that touch its slice.
// The other sums are exchanged by pushing every CTA's partial sums to all
// CTAs, which add them in rank order: all CTAs hold the same scalars and take
// the same branches.  Four cluster barriers an iteration: p; p.q; r.r
// with S^T r and Y^T r; r.z.
// The compact L-BFGS form is applied as one 2k x 2k matrix, formed when the
// pairs are chosen, instead of two triangular solves by one thread.
//
// Bound by latency (barriers and short dependent chains).  One CTA took
// FP64-pipe time instead: on 26 x 26 nodes with 20 pairs half of it in the
// minimal-surface elements, most of the rest in the 2 x 40 dots and updates and
// the serial solves.  The 101^2 minimal-surface solve with the paper's settings
// went from 313.6 ms (89 % in this solver) to 60.6 ms.
#include <cooperative_groups.h>

#include "coarse.cuh"
#include "coarse_elem.cuh"
#include "reduce.cuh"
#include "stencil.cuh"

namespace jfnk {

namespace cg = cooperative_groups;

constexpr int kCgThreads = 512;
constexpr int kCgMaxCtas = 8;
constexpr int kMaxShiftCalls = 30;
constexpr int kCgVals = 2 * kMaxLbfgsPairs + 4;  // sums exchanged at once

struct CgOut {
    double lam_c;  // Rayleigh quotient at negative curvature, else 0
    int its;
    int fd;        // FD actions (level-0 gradient evaluations)
    int negcurv;
};

// Shared memory of a CTA: doubles first, then the T arrays.
struct CgLayout {
    int sl;                                   // slice length
    size_t slots, tot, mat, coef, scal, part, step;  // doubles
    size_t x, r, z, p, q, x0, ax, S, Y, xw, ec, mask;
    size_t bytes;
};
__host__ __device__ inline CgLayout cg_layout(int N, int ne, int npe, int ctas, size_t esz) {
    CgLayout l;
    const int k = kMaxLbfgsPairs;  // (the pairs kept may come from a call with other options)
    l.sl = (N + ctas - 1) / ctas;
    size_t o = 0;
    auto take = [&](size_t count, size_t size) {
        o = (o + 15) & ~size_t(15);
        const size_t at = o;
        o += count * size;
        return at;
    };
    l.slots = take((size_t)2 * ctas * kCgVals, 8);
    l.tot = take(kCgVals, 8);
    l.mat = take((size_t)4 * k * k, 8);
    l.coef = take(2 * k, 8);
    l.scal = take(8, 8);
    l.part = take(kCgThreads / 32, 8);
    l.step = take(1, sizeof(EpsSlot));
    size_t* v[] = {&l.x, &l.r, &l.z, &l.p, &l.q, &l.ax};
    for (size_t* a : v) *a = take(l.sl, esz);
    l.x0 = take(N, esz);
    l.S = take((size_t)k * l.sl, esz);
    l.Y = take((size_t)k * l.sl, esz);
    l.xw = take(N, esz);
    l.ec = take((size_t)ne * npe, esz);
    l.mask = take(l.sl, 1);
    l.bytes = o;
    return l;
}

template <typename T, Prob P>
struct CgCta {
    const CoarseArgs<T>& a;
    cg::cluster_group cluster;
    const CgLayout& l;
    const CoarseElem<T, P> ce;
    unsigned char* sm;
    int rank, ctas, N, i0, n;  // owned entries [i0, i0 + n)
    int buf = 0;               // slot buffer of the next exchange
    double gamma = 1.0;
    EpsPre pre;

    __device__ CgCta(const CoarseArgs<T>& args, const CgLayout& lay, unsigned char* smem)
        : a(args), cluster(cg::this_cluster()), l(lay), ce(args.lh), sm(smem) {
        rank = (int)cluster.block_rank();
        ctas = (int)cluster.num_blocks();
        N = (int)a.g.size;
        i0 = rank * l.sl;
        n = max(0, min(l.sl, N - i0));
        const EpsParams ep = {a.eps_mode, a.n_unknowns, a.xstat};
        pre = eps_pre(ep);
    }
    __device__ double* dbl(size_t o) const { return reinterpret_cast<double*>(sm + o); }
    __device__ T* vec(size_t o) const { return reinterpret_cast<T*>(sm + o); }
    __device__ bool inner(int i) const { return sm[l.mask + i] != 0; }
    __device__ double& scal(int i) const { return dbl(l.scal)[i]; }
    __device__ EpsSlot& slot() const { return *reinterpret_cast<EpsSlot*>(sm + l.step); }

    // sum v of this CTA's slice of u . w, by one warp, to every CTA
    __device__ void dot_push(int v, const T* u, const T* w) {
        const int lane = threadIdx.x & 31;
        double d = 0.0;
        for (int i = lane; i < n; i += 32) d += (double)u[i] * (double)w[i];
        d = warp_sum(d);
        if (lane < ctas) {
            double* s = dbl(l.slots) + ((size_t)buf * ctas + rank) * kCgVals + v;
            *cluster.map_shared_rank(s, lane) = d;
        }
    }
    // totals of the nv sums pushed since the last exchange, in every CTA;
    // warp 0 sums them, `f` runs in its lane 0 on the totals
    template <typename F>
    __device__ void exchange(int nv, F f) {
        cluster.sync();
        if (threadIdx.x < 32) {
            const double* s = dbl(l.slots) + (size_t)buf * ctas * kCgVals;
            for (int v = threadIdx.x; v < nv; v += 32) {
                double t = 0.0;
                for (int c = 0; c < ctas; ++c) t += s[c * kCgVals + v];
                dbl(l.tot)[v] = t;
            }
            __syncwarp();
            if (threadIdx.x == 0) f(dbl(l.tot));
        }
        buf ^= 1;
        __syncthreads();
    }

    // FD step for a direction of squared norm pp (0: none)
    __device__ void step(double pp) { set_eps_slot(&slot(), pre, pp, false, nullptr); }
    // q = A_s p = (A(x_0 + eps p) - A(x_0)) / eps - shift p on the slice; p.p in
    // scal 4, the step in the slot
    __device__ void apply(const T* p, double shift) {
        const Grid& g = a.g;
        T* q = vec(l.q);
        T* xw = vec(l.xw);
        for (int t = threadIdx.x; t < n * ctas; t += blockDim.x) {
            const int c = t / n, i = t - c * n;
            *cluster.map_shared_rank(xw + i0 + i, c) = p[i];
        }
        cluster.sync();
        // every CTA has all of p and sums p.p in the same order
        double d = 0.0;
        for (int i = threadIdx.x; i < N; i += blockDim.x) d += (double)xw[i] * (double)xw[i];
        d = warp_sum(d);
        if ((threadIdx.x & 31) == 0) dbl(l.part)[threadIdx.x >> 5] = d;
        __syncthreads();
        if (threadIdx.x < 32) {
            d = warp_sum(threadIdx.x < kCgThreads / 32 ? dbl(l.part)[threadIdx.x] : 0.0);
            if (threadIdx.x == 0) {
                scal(4) = d;
                step(d);
            }
        }
        __syncthreads();
        const T eps = (T)slot().e, inv = (T)slot().inv, sh = (T)shift;
        if (!(slot().e > 0.0)) {
            for (int i = threadIdx.x; i < n; i += blockDim.x) q[i] = T(0);
            __syncthreads();
            return;
        }
        for (int i = threadIdx.x; i < N; i += blockDim.x) xw[i] = vec(l.x0)[i] + eps * xw[i];
        __syncthreads();
        // elements touching the nodes of the slice
        T* ec = vec(l.ec);
        const int nc = g.nc;
        const int va = i0 / nc, vb = n > 0 ? (i0 + n - 1) / nc : -1;  // owned nodes
        const int ex = g.beam ? 10 * g.n : g.n, ey = g.n, npe = coarse_npe(g);
        const int nxy = g.nx * g.ny;
        if (is_2d(P)) {
            const int ya = max(0, va / g.nx - 1), yb = min(ey - 1, vb / g.nx);
            for (int t = threadIdx.x; n > 0 && t < (yb - ya + 1) * ex; t += blockDim.x) {
                const int y = ya + t / ex, x = t % ex, v = y * g.nx + x;
                if (v + g.nx + 1 < va || v > vb) continue;
                coarse_element<T, P>(g, xw, x, y, 0, T(1), a.lh, ce, ec + (y * ex + x) * npe);
            }
        } else {
            const int za = max(0, va / nxy - 1), zb = min(ey - 1, vb / nxy);
            for (int t = threadIdx.x; n > 0 && t < (zb - za + 1) * ex * ey; t += blockDim.x) {
                const int z = za + t / (ex * ey), y = (t / ex) % ey, x = t % ex, v = z * nxy + y * g.nx + x;
                // its corners are v, v + 1, and those one row and one plane up
                auto hits = [&](int u) { return u + 1 >= va && u <= vb; };
                if (!hits(v) && !hits(v + g.nx) && !hits(v + nxy) && !hits(v + nxy + g.nx)) continue;
                const int e = (z * ey + y) * ex + x;
                coarse_element<T, P>(g, xw, x, y, z, P == Prob::NDK3 ? a.kappa[e] : T(1), a.lh, ce, ec + e * npe);
            }
        }
        __syncthreads();
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            T acc = T(0);
            if (inner(i)) {
                const int node = (i0 + i) / nc, comp = (i0 + i) - node * nc;
                const int X = node % g.nx, Y = (node / g.nx) % g.ny, Z = node / nxy;
#pragma unroll
                for (int c = 0; c < (is_2d(P) ? 4 : 8); ++c) {
                    const int xe = X - (c & 1), ye = Y - ((c >> 1) & 1), ze = Z - (c >> 2);
                    if (xe < 0 || xe >= ex || ye < 0 || ye >= ey || ze < 0 || (!is_2d(P) && ze >= ey)) continue;
                    acc += ec[((ze * ey + ye) * ex + xe) * npe + c * nc + comp];
                }
                acc = (acc * a.node_scale - vec(l.ax)[i]) * inv - sh * p[i];
            }
            q[i] = acc;
        }
        __syncthreads();
    }

    // z = H r on the slice from the sums S^T r, Y^T r in tot[1..]
    __device__ void precond(int k) {
        const T* r = vec(l.r);
        T* z = vec(l.z);
        if (k <= 0) {
            for (int i = threadIdx.x; i < n; i += blockDim.x) z[i] = r[i];
            __syncthreads();
            return;
        }
        // coef = C dots, 8 lanes a row
        const double* C = dbl(l.mat);
        const double* d = dbl(l.tot) + 1;
        const int sub = threadIdx.x & 7;
        for (int row = threadIdx.x >> 3; row < ((2 * k + 3) & ~3); row += blockDim.x >> 3) {
            double s = 0.0;
            if (row < 2 * k)
                for (int j = sub; j < 2 * k; j += 8) s += C[row * 2 * k + j] * d[j];
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (sub == 0 && row < 2 * k) dbl(l.coef)[row] = s;
        }
        __syncthreads();
        const double* co = dbl(l.coef);
        const T *S = vec(l.S), *Y = vec(l.Y);
        const int part = threadIdx.x & 3;  // 4 lanes an entry
        for (int i = threadIdx.x >> 2; i < ((n + 7) & ~7); i += blockDim.x >> 2) {
            double s = 0.0;
            if (i < n) {
                for (int j = part; j < k; j += 4)
                    s += co[j] * (double)S[j * l.sl + i] + co[k + j] * (double)Y[j * l.sl + i];
            }
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            s += __shfl_xor_sync(0xffffffffu, s, 2);
            if (part == 0 && i < n) z[i] = inner(i) ? (T)(gamma * (double)r[i] + s) : T(0);
        }
        __syncthreads();
    }

    // CG(s_0, x_0, F(x_0), r_0, lambda_c+) of Alg. 1
    __device__ CgOut run(double shift, bool warm, int k, bool collect, double target) {
        T *x = vec(l.x), *r = vec(l.r), *z = vec(l.z), *p = vec(l.p), *q = vec(l.q);
        const T *S = vec(l.S), *Y = vec(l.Y);
        const int tid = threadIdx.x, wid = tid >> 5, nw = blockDim.x >> 5;
        CgOut o = {0.0, 0, 0, 0};
        if (warm) {
            apply(x, shift);
            o.fd++;
        }
        for (int i = tid; i < n; i += blockDim.x) r[i] = inner(i) ? (warm ? a.b[i0 + i] - q[i] : a.b[i0 + i]) : T(0);
        __syncthreads();
        // r.r, S^T r, Y^T r
        auto residual_sums = [&]() {
            for (int v = wid; v <= 2 * k; v += nw)
                dot_push(v, r, v == 0 ? r : v <= k ? S + (v - 1) * l.sl : Y + (v - 1 - k) * l.sl);
            exchange(1 + 2 * k, [&](double* t) { scal(2) = sqrt(t[0]); });
        };
        residual_sums();
        double res = scal(2);
        if (!(res > 0.0) || res <= target || !isfinite(res)) return o;
        precond(k);
        for (int i = tid; i < n; i += blockDim.x) p[i] = T(0);
        __syncthreads();
        if (wid == 0) dot_push(0, r, z);
        exchange(1, [&](double* t) {
            scal(3) = t[0];  // r.z
            scal(5) = 0.0;   // beta
        });
        for (int it = 1; it <= a.maxit; ++it) {
            const T beta = (T)scal(5);
            for (int i = tid; i < n; i += blockDim.x) p[i] = z[i] + beta * p[i];
            __syncthreads();
            apply(p, shift);
            o.fd++;
            o.its = it;
            if (wid == 0) dot_push(0, p, q);
            exchange(1, [&](double* t) { scal(6) = scal(3) / t[0]; });
            const double pq = dbl(l.tot)[0];
            if (!isfinite(pq)) return o;
            if (pq <= 0.0) {
                const double pp = scal(4);
                o.lam_c = pp > 0.0 ? pq / pp : 0.0;
                o.negcurv = 1;
                return o;
            }
            const T al = (T)scal(6);
            for (int i = tid; i < n; i += blockDim.x) {
                if (collect) {
                    a.S_all[(long long)(it - 1) * N + i0 + i] = al * p[i];
                    a.Y_all[(long long)(it - 1) * N + i0 + i] = al * q[i];
                }
                x[i] += al * p[i];
                r[i] -= al * q[i];
            }
            if (collect && tid == 0 && rank == 0) a.lb->collected = it;
            __syncthreads();
            residual_sums();
            res = scal(2);
            if (res <= target || !isfinite(res)) return o;
            precond(k);
            if (wid == 0) dot_push(0, r, z);
            exchange(1, [&](double* t) {
                scal(5) = t[0] / scal(3);
                scal(3) = t[0];
            });
        }
        return o;
    }

    // keep m of the collected pairs (uniform sampling) and set up the compact form
    __device__ void build() {
        const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5;
        LbfgsState* lb = a.lb;
        cluster.sync();  // every CTA's part of the collected pairs
        const int kall = __ldcg(&lb->collected);
        const int m = min(a.m_pairs, kMaxLbfgsPairs);
        const int k = min(kall, m);
        for (int j = 0; j < k; ++j) {
            const long long src = (kall > m) ? ((long long)j * kall) / m : j;
            for (int i = i0 + tid; i < i0 + n; i += blockDim.x) {
                a.S[(long long)j * N + i] = __ldcg(&a.S_all[src * N + i]);
                a.Y[(long long)j * N + i] = __ldcg(&a.Y_all[src * N + i]);
            }
        }
        cluster.sync();
        // R_ij = s_i.y_j (i <= j), YtY_ij = y_i.y_j, the pairs (i, j) dealt over the cluster's warps
        for (int q = rank * nw + wid; q < 2 * k * k; q += ctas * nw) {
            const int which = q / (k * k), ij = q % (k * k), i = ij / k, j = ij % k;
            const T* u = (which == 0) ? a.S + (long long)i * N : a.Y + (long long)i * N;
            const T* v = a.Y + (long long)j * N;
            double d = 0.0;
            for (int t = lane; t < N; t += 32) d += (double)__ldcg(&u[t]) * (double)__ldcg(&v[t]);
            d = warp_sum(d);
            if (lane == 0) {
                if (which == 0)
                    lb->R[i * kMaxLbfgsPairs + j] = (i <= j) ? d : 0.0;
                else
                    lb->YtY[i * kMaxLbfgsPairs + j] = d;
            }
        }
        cluster.sync();
        if (rank == 0 && tid == 0) {
            bool ok = k > 0;
            for (int i = 0; i < k; ++i) ok = ok && __ldcg(&lb->R[i * kMaxLbfgsPairs + i]) > 0.0;
            const int last = (k - 1) * kMaxLbfgsPairs + (k - 1);
            const double yy = k > 0 ? __ldcg(&lb->YtY[last]) : 0.0;
            lb->gamma = (ok && yy > 0.0) ? __ldcg(&lb->R[last]) / yy : 1.0;
            lb->count = (ok && yy > 0.0) ? k : 0;
        }
        cluster.sync();
    }

    // this CTA's slice of the kept pairs and the matrix of the compact form,
    //   C = [R^-T (D + gamma Y^T Y) R^-1, -gamma R^-T; -gamma R^-1, 0],
    // column c of it by thread c (H r = gamma r + [S Y] C [S^T r; Y^T r])
    __device__ void load_pairs(int k) {
        const int tid = threadIdx.x;
        const LbfgsState* lb = a.lb;
        T *S = vec(l.S), *Y = vec(l.Y);
        for (int t = tid; t < k * n; t += blockDim.x) {
            const int j = t / n, i = t - j * n;
            S[j * l.sl + i] = __ldcg(&a.S[(long long)j * N + i0 + i]);
            Y[j * l.sl + i] = __ldcg(&a.Y[(long long)j * N + i0 + i]);
        }
        double* C = dbl(l.mat);
        gamma = __ldcg(&lb->gamma);
        const double gam = gamma;
        constexpr int K = kMaxLbfgsPairs;
        auto R = [&](int i, int j) { return __ldcg(&lb->R[i * K + j]); };
        if (tid < 2 * k) {
            double t[K], v[K];
            const int c = tid < k ? tid : tid - k;
            if (tid < k) {
                // t = R^-1 e_c; v = (D + gamma Y^T Y) t
                for (int i = k - 1; i >= 0; --i) {
                    double s = i == c ? 1.0 : 0.0;
                    for (int j = i + 1; j < k; ++j) s -= R(i, j) * t[j];
                    t[i] = s / R(i, i);
                }
                for (int i = 0; i < k; ++i) {
                    double s = R(i, i) * t[i];
                    for (int j = 0; j < k; ++j) s += gam * __ldcg(&lb->YtY[i * K + j]) * t[j];
                    v[i] = s;
                }
            } else {
                for (int i = 0; i < k; ++i) {
                    t[i] = 0.0;
                    v[i] = i == c ? -gam : 0.0;
                }
            }
            // R^-T v
            for (int i = 0; i < k; ++i) {
                double s = v[i];
                for (int j = 0; j < i; ++j) s -= R(j, i) * v[j];
                v[i] = s / R(i, i);
            }
            for (int i = 0; i < k; ++i) {
                C[i * 2 * k + tid] = v[i];
                C[(k + i) * 2 * k + tid] = -gam * t[i];
            }
        }
        __syncthreads();
    }
};

template <typename T, Prob P>
__global__ void __launch_bounds__(kCgThreads) coarse_cgqn_kernel(const CoarseArgs<T> a, const CgLayout l) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    CgCta<T, P> c(a, l, smem_raw);
    const int tid = threadIdx.x;
    for (int i = tid; i < c.n; i += blockDim.x) {
        const bool in = coarse_inner(a.g, c.i0 + i);
        smem_raw[l.mask + i] = in ? 1 : 0;
        c.vec(l.x)[i] = T(0);
        c.vec(l.ax)[i] = a.Ax[c.i0 + i];
        c.vec(l.z)[i] = in ? a.b[c.i0 + i] : T(0);
    }
    for (int i = tid; i < c.N; i += blockDim.x) c.vec(l.x0)[i] = a.x[i];
    const int count = __ldcg(&a.lb->count);
    const bool collect = count < 0;
    int k = collect ? 0 : count;
    if (k > 0) c.load_pairs(k);
    __syncthreads();
    c.cluster.sync();  // every CTA of the cluster runs before its memory is written
    if (tid < 32) c.dot_push(0, c.vec(l.z), c.vec(l.z));
    c.exchange(1, [&](double* t) { c.scal(7) = sqrt(t[0]); });
    const double target = a.tol_abs ? a.tol : a.tol * c.scal(7);
    long long fd = 0;
    int negc = 0, nshift = 0;
    double shift = 0.0;
    CgOut o = c.run(shift, false, k, collect, target);
    fd += o.fd;
    negc += o.negcurv;
    if (collect) {
        c.build();
        k = __ldcg(&a.lb->count);
        if (k > 0 && o.lam_c < 0.0) c.load_pairs(k);
    }
    while (o.lam_c < 0.0 && nshift < kMaxShiftCalls) {
        shift = a.shift_gamma * fmin(o.lam_c, shift);
        ++nshift;
        o = c.run(shift, true, k, false, target);
        fd += o.fd;
        negc += o.negcurv;
    }
    for (int i = tid; i < c.n; i += blockDim.x) a.s[c.i0 + i] = c.inner(i) ? c.vec(l.x)[i] : T(0);
    if (tid == 0 && c.rank == 0) {
        if (a.iters) *a.iters += fd;
        a.lb->shifts += nshift;
        a.lb->negcurv += negc;
    }
    c.cluster.sync();  // no CTA leaves while another may still write to it
}

template <typename T, Prob P>
static jfnk_status launch_cgqn_p(const CoarseArgs<T>& a, cudaStream_t st) {
    const int N = (int)a.g.size, ne = (int)a.g.elements(), npe = coarse_npe(a.g);
    // about 64 entries a CTA, at most 8 CTAs (the portable cluster size)
    const int ctas = N <= 64 ? 1 : (N + 63) / 64 < kCgMaxCtas ? (N + 63) / 64 : kCgMaxCtas;
    const CgLayout l = cg_layout(N, ne, npe, ctas, sizeof(T));
    if (l.bytes > 200 * 1024) {
        set_error("coarse solver shared memory %zu too large", l.bytes);
        return JFNK_ERR_INVALID_ARG;
    }
    auto kernel = coarse_cgqn_kernel<T, P>;
    JFNK_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)l.bytes));
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = ctas;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(kCgThreads);
    cfg.dynamicSmemBytes = l.bytes;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    JFNK_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, a, l));
    JFNK_LAUNCH_CHECK();
    return JFNK_OK;
}

template <typename T>
jfnk_status launch_coarse_cgqn(Prob prob, const CoarseArgs<T>& a, cudaStream_t st) {
    if (a.adjoint) {
        set_error("the CG-QN coarse solver is implemented for the forward operator");
        return JFNK_ERR_NOT_IMPLEMENTED;
    }
    if (!a.lb || !a.S_all || !a.Y_all || !a.S || !a.Y || a.m_pairs < 1 || a.m_pairs > kMaxLbfgsPairs) {
        set_error("CG-QN coarse solver: workspace not laid out for it, or 1 <= pairs <= %d violated", kMaxLbfgsPairs);
        return JFNK_ERR_WORKSPACE;
    }
    switch (prob) {
        case Prob::BRATU2: return launch_cgqn_p<T, Prob::BRATU2>(a, st);
        case Prob::MINSURF2: return launch_cgqn_p<T, Prob::MINSURF2>(a, st);
        case Prob::BEAM3: return launch_cgqn_p<T, Prob::BEAM3>(a, st);
        case Prob::ND3: return launch_cgqn_p<T, Prob::ND3>(a, st);
        case Prob::NDK3: return launch_cgqn_p<T, Prob::NDK3>(a, st);
    }
    set_error("unknown problem kind");
    return JFNK_ERR_INVALID_ARG;
}
template jfnk_status launch_coarse_cgqn<float>(Prob, const CoarseArgs<float>&, cudaStream_t);
template jfnk_status launch_coarse_cgqn<double>(Prob, const CoarseArgs<double>&, cudaStream_t);

}  // namespace jfnk
