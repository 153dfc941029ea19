// Batched kernels: one launch applies a level operation to every active
// instance of a batch of independent problems of uneven sizes.  Each CTA
// finds its instance in a segment list and reads that instance's operands
// from descriptor arrays in device memory; reductions complete per instance
// (each instance's CTAs form one segment of the last-block reduction).
#pragma once
#include "common.cuh"
#include "stencil.cuh"

namespace jfnk {

// One instance's CTAs in a batched launch: consecutive blocks from `first`.  A CTA
// finds its instance among the segments (sorted by first) with one load a lane
// and a ballot per 32 segments, so that a launch's work list is one entry per
// instance and not one per CTA.
struct BSeg {
    int first, nblk;
    int strips, rows;  // 2D kernel: strips of node columns, node rows a CTA (stencil_fx2d.cuh)
};

// per-instance operands of a batched vector operation
struct BVec {
    Grid g;            // grid of x / y
    Grid gc;           // coarse grid (transfers)
    void* y;           // output
    const void* x;     // input
    const void* x2;    // second input
    void* y2;          // second output
    double a, b;       // scalars
    const double* dsc; // device scalar operand
    double* out;       // reduction result(s)
    EpsSlot* slot;     // FD step produced by a norm
    EpsParams ep;
    const ChebTable* cheb;
    double* partials;  // this instance's reduction scratch
    unsigned int* counter;
    long long ld;      // leading dimension of a vector block (FGMRES bases)
    int m;             // number of vectors in a block operation
    int what;          // op detail (statistic kind, projection flag, ...)
    uint64_t key;      // SplitMix64 stream key
};

enum class BOp : int {
    CAST_D2T = 0,    // y(T) = x(double)
    CAST_T2D = 1,    // y(double) = x(T)
    COPY_T = 2,      // y = x
    AXPBY_D = 3,     // y = a x + b y              (double)
    ADDSC_D = 4,     // y = x + a x2              (double)
    SCALE_INV_T = 5, // y = x / *dsc (0 if *dsc == 0)
    STAT = 6,        // out = sum|x| (what 0) or ||x|| (what 1), interior; slot (if set) = FD step
    CHEB_START = 7,  // y = r = b(x) interior, y2 = d = b / theta, s(x2 as output) = 0; ||d|| -> slot
    RESTRICT = 8,    // y(gc) = I^T x (what 1: projection 2^-d, boundary injection)
    PROLONG_ADD = 9, // y += I x(gc)
    SPLITMIX = 10,   // y = uniform [-1,1) start vector from key (interior)
    MDOT = 11,       // out[k] = <x, x2 + k ld>, k < m   (double)
    MAXPY_SUB = 12,  // y -= sum_k out[k] (x2 + k ld)   (double; out read as coefficients)
    COMBINE_T = 13,  // y(double) += sum_k dsc[k] (x(T) + k ld)
    CAST_SCALE_INT_D = 14,  // y(double) = a x(double) on interior, 0 on the boundary
};

// Tiny per-instance scalar kernels (one thread per instance)
enum class BScalar : int {
    CHEB_TABLE = 1,  // cheb table from *x with [a, b] and degree m
    SET_EPS = 2,     // slot from a
    GATHER = 3,      // out[0..m) = x[0..m); out[kGatherIters] = *x2 (bits); out[kGatherStatus] = *status
};
constexpr int kGatherIters = JFNK_MAX_LEVELS, kGatherStatus = JFNK_MAX_LEVELS + 1;
struct BScal {
    double* out;
    const double* x;
    const double* x2;
    double a, b;
    int m;
    ChebTable* cheb;
    EpsSlot* slot;
    int* status;
};

// `blocks` CTAs of bx threads over `count` instances
template <typename T>
jfnk_status launch_stencil2d_batched(Mode mode, const StencilArgs<T>* dev_args, const BSeg* dev_segs, int count,
                                     int blocks, int bx, cudaStream_t st);

template <typename T>
jfnk_status launch_bvec(BOp op, const BVec* dev_desc, const BSeg* dev_segs, int count, int blocks, cudaStream_t st);

jfnk_status launch_bscalar(BScalar op, const BScal* dev_desc, int count, cudaStream_t st);

}  // namespace jfnk
