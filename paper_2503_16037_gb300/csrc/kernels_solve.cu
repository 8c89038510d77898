// Solver kernels for (I - K) x = s (Eq. flux_system of Mikkonen et al.;
// the Neumann / source iteration is the series of Eq. fs_sum).
//
// The sweeps walk rows of receivers (K in CSR order by row) in groups of 128
// rows; the column of each slot comes from the row template of the row's
// layer instead of a stored index, so only the 4-byte values stream.
// Reductions are deterministic: fixed grids, fixed per-block order,
// fixed-order trees.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "kern.h"
#include "stage.cuh"

namespace tk {

// ---- Row-group kernels.  One pass over K does one of the operations below
// (an "Op"): it accumulates, for each row of a group, the products of the
// row's values with the source values it gathers, and finishes the row
// (combination of the warps' partial sums in a fixed order, the row update,
// per-group partial sums of squares).  The plain driver runs one block of W
// warps per group and reads the values directly; for FP32 ops that gather
// from FP32 vectors it first copies the group's source rows into a
// shared-memory tile (k_tile); the pipelined driver (k_pipe) streams the
// values through shared memory.  Source values are gathered from haloed
// vectors (the template offset is the only index arithmetic), and every row
// result is stored with its halo copies.

// Op interface (both drivers): A / NA: accumulator type and words per lane;
// kPart: the op writes per-row-block partial sums part[4 gi + k]; Pre: the
// epilogue inputs of one row, loaded when a group starts (pre) so that their
// latency hides behind the group's slots; slot / add: per-slot constants and
// the accumulation of one value times one gathered source value;
// combine_row: the words of row k summed over the W warps in a fixed order;
// finish_row: the row update, returning the row's share of the partial sum.

// The refinement update x += d (with the FP32-pair split of x when xh is
// set), done row by row in the epilogue of the pass that produces d
// (x == nullptr: none); the same arithmetic as k_update_x.
struct XUpd {
    double *x = nullptr;
    float *xh = nullptr, *xl = nullptr;
    template <typename T>
    __device__ __forceinline__ void apply(const GroupRows &G, int k, T d) const {
        if (x == nullptr) return;
        const double v = x[G.rp[k]] + (double)d;
        store_h(x, G, k, v);
        if (xh) {
            const float h = (float)v;
            store_h(xh, G, k, h);
            store_h(xl, G, k, (float)(v - (double)h));
        }
    }
};

// MODE 0: y = b + K x (b may be null); MODE 1: y = x - K x
template <typename T, int MODE>
struct OpSpmv {
    using A = T;
    static constexpr int NA = 4;
    static constexpr bool kPart = false;
    struct Pre {
        T u;
    };
    const T *x, *b;
    T *y;
    static constexpr int kTile = sizeof(T) == 4 ? 1 : 0;
    __device__ __forceinline__ const T *gsrc(int) const { return x; }
    __device__ __forceinline__ void add_t(A *a, int k, T v, const T *s, int, NoSlot) const { a[k] += v * s[0]; }
    __device__ __forceinline__ NoSlot slot(const GraphP &, int) const { return NoSlot(); }
    __device__ __forceinline__ void add(A *a, int k, T v, int j, NoSlot) const { a[k] += v * __ldg(x + j); }
    __device__ __forceinline__ Pre pre(const GroupRows &G, int k) const {
        Pre p;
        p.u = MODE == 0 ? (b ? b[G.rp[k]] : T(0)) : x[G.rp[k]];
        return p;
    }
    template <int W>
    __device__ __forceinline__ static void combine_row(const A (*sh)[NA][32], int lane, int k, A *a) {
        sum_word<W, A, NA>(sh, lane, k, a);
    }
    __device__ __forceinline__ double finish_row(const GroupRows &G, int k, const A *a, const Pre &p) const {
        store_h(y, G, k, MODE == 0 ? p.u + a[k] : p.u - a[k]);
        return 0.0;
    }
};

// r = s - x + K x with FP64 x and FP64 accumulation; partial sums of r^2
template <typename T>
struct OpResid64 {
    using A = double;
    static constexpr int NA = 4;
    static constexpr bool kPart = true;
    struct Pre {
        double s, x;
    };
    const T *s;
    const double *x;
    double *r, *part;
    __device__ __forceinline__ NoSlot slot(const GraphP &, int) const { return NoSlot(); }
    __device__ __forceinline__ void add(A *a, int k, T v, int j, NoSlot) const { a[k] += (double)v * __ldg(x + j); }
    __device__ __forceinline__ Pre pre(const GroupRows &G, int k) const {
        Pre p;
        p.s = (double)s[G.row[k]];
        p.x = x[G.rp[k]];
        return p;
    }
    template <int W>
    __device__ __forceinline__ static void combine_row(const A (*sh)[NA][32], int lane, int k, A *a) {
        sum_word<W, A, NA>(sh, lane, k, a);
    }
    __device__ __forceinline__ double finish_row(const GroupRows &G, int k, const A *a, const Pre &p) const {
        const double vv = p.s - p.x + a[k];
        store_h(r, G, k, vv);
        return vv * vv;
    }
};

// Neumann sweep y = b + K x with partial sums of (y - x)^2
template <typename T>
struct OpSweepPow {
    using A = T;
    static constexpr int NA = 4;
    static constexpr bool kPart = true;
    struct Pre {
        T b, x;
    };
    const T *x, *b;
    T *y;
    double *part;
    XUpd xu;
    static constexpr int kTile = sizeof(T) == 4 ? 1 : 0;
    __device__ __forceinline__ const T *gsrc(int) const { return x; }
    __device__ __forceinline__ void add_t(A *a, int k, T v, const T *s, int, NoSlot) const { a[k] += v * s[0]; }
    __device__ __forceinline__ NoSlot slot(const GraphP &, int) const { return NoSlot(); }
    __device__ __forceinline__ void add(A *a, int k, T v, int j, NoSlot) const { a[k] += v * __ldg(x + j); }
    __device__ __forceinline__ Pre pre(const GroupRows &G, int k) const {
        Pre p;
        p.b = b[G.rp[k]];
        p.x = x[G.rp[k]];
        return p;
    }
    template <int W>
    __device__ __forceinline__ static void combine_row(const A (*sh)[NA][32], int lane, int k, A *a) {
        sum_word<W, A, NA>(sh, lane, k, a);
    }
    __device__ __forceinline__ double finish_row(const GroupRows &G, int k, const A *a, const Pre &p) const {
        const T vv = p.b + a[k];
        const T dd = vv - p.x;
        store_h(y, G, k, vv);
        xu.apply(G, k, vv);
        return (double)(dd * dd);
    }
};

// The two products of a BiCGStab step: y = x - K x with its dot products.
// ND 1: r0.y; ND 5: y.x, y.y, r0.x, r0.y, x.x
template <typename T, int ND>
struct OpBi {
    using A = T;
    static constexpr int NA = 4;
    static constexpr bool kPart = false;
    static constexpr int kDots = ND;
    struct Pre {
        T u, q0;
    };
    const T *x, *r0;
    T *y;
    double *part;
    size_t pstride;
    const BiState<T> *st;
    static constexpr int kTile = sizeof(T) == 4 ? 1 : 0;
    __device__ __forceinline__ bool skip() const { return *(volatile const int *)&st->done != 0; }
    __device__ __forceinline__ const T *gsrc(int) const { return x; }
    __device__ __forceinline__ void add_t(A *a, int k, T v, const T *s, int, NoSlot) const { a[k] += v * s[0]; }
    __device__ __forceinline__ NoSlot slot(const GraphP &, int) const { return NoSlot(); }
    __device__ __forceinline__ void add(A *a, int k, T v, int j, NoSlot) const { a[k] += v * __ldg(x + j); }
    __device__ __forceinline__ Pre pre(const GroupRows &G, int k) const {
        Pre p;
        p.u = x[G.rp[k]];
        p.q0 = r0[G.rp[k]];
        return p;
    }
    template <int W>
    __device__ __forceinline__ static void combine_row(const A (*sh)[NA][32], int lane, int k, A *a) {
        sum_word<W, A, NA>(sh, lane, k, a);
    }
    __device__ __forceinline__ void finish_dots(const GroupRows &G, int k, const A *a, const Pre &p, Dot<T> *d) const {
        const T v = p.u - a[k];
        store_h(y, G, k, v);
        if constexpr (ND == 1) {
            d[0].add(p.q0, v);
        } else {
            d[0].add(v, p.u);
            d[1].add(v, v);
            d[2].add(p.q0, p.u);
            d[3].add(p.q0, v);
            d[4].add(p.u, p.u);
        }
    }
};

// One Chebyshev step on (I - K) d = r0 (three-term form):
//   q = K p;  r <- r - p + q;  d <- d + p;  p' = c1 p + c2 r
template <typename T>
struct OpCheb {
    using A = T;
    static constexpr int NA = 4;
    static constexpr bool kPart = false;
    struct Pre {
        T p, r, d;
    };
    const T *p;
    T *r, *d, *pn;
    T c1, c2;
    XUpd xu;
    static constexpr int kTile = sizeof(T) == 4 ? 1 : 0;
    __device__ __forceinline__ const T *gsrc(int) const { return p; }
    __device__ __forceinline__ void add_t(A *a, int k, T v, const T *s, int, NoSlot) const { a[k] += v * s[0]; }
    __device__ __forceinline__ NoSlot slot(const GraphP &, int) const { return NoSlot(); }
    __device__ __forceinline__ void add(A *a, int k, T v, int j, NoSlot) const { a[k] += v * __ldg(p + j); }
    __device__ __forceinline__ Pre pre(const GroupRows &G, int k) const {
        const int ip = G.rp[k];
        Pre q;
        q.p = p[ip];
        q.r = r[ip];
        q.d = d[ip];
        return q;
    }
    template <int W>
    __device__ __forceinline__ static void combine_row(const A (*sh)[NA][32], int lane, int k, A *a) {
        sum_word<W, A, NA>(sh, lane, k, a);
    }
    __device__ __forceinline__ double finish_row(const GroupRows &G, int k, const A *a, const Pre &q) const {
        const T rr = q.r - q.p + a[k];
        store_h(r, G, k, rr);
        const T dn = q.d + q.p;
        store_h(d, G, k, dn);
        xu.apply(G, k, dn);
        store_h(pn, G, k, c1 * q.p + c2 * rr);
        return 0.0;
    }
};

// ---- residual in double-single arithmetic (pairs of FP32 numbers).  x is
// held as x_hi + x_lo (x_hi = fl32(x), x_lo = fl32(x - x_hi)); each product
// v x_hi is split exactly into p + e with an FMA (two-product), the p are
// summed with Knuth's two-sum and all low-order parts are gathered in a
// second FP32 accumulator.  The row sum so obtained carries a relative error
// of order 2^-48 per term instead of 2^-24.
// (explicitly rounded operations: none of them may be contracted into an FMA)
__device__ __forceinline__ void ds_add_prod(float &hi, float &lo, float v, float xh, float xl) {
    const float p = __fmul_rn(v, xh);
    const float e = fmaf(v, xh, -p);
    const float s = __fadd_rn(hi, p);
    const float bb = __fsub_rn(s, hi);
    const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(p, bb));
    hi = s;
    lo = __fadd_rn(lo, __fadd_rn(__fadd_rn(err, e), __fmul_rn(v, xl)));
}

// r = s - x + K x with K x summed in FP32 pairs (a[k]: high part, a[4 + k]: low part)
struct OpResidDS {
    using A = float;
    static constexpr int NA = 8;
    static constexpr bool kPart = true;
    struct Pre {
        double s, x;
    };
    const float *s;
    const double *x;
    const float *xh, *xl;
    double *r, *part;
    __device__ __forceinline__ NoSlot slot(const GraphP &, int) const { return NoSlot(); }
    __device__ __forceinline__ void add(A *a, int k, float v, int j, NoSlot) const {
        ds_add_prod(a[k], a[4 + k], v, __ldg(xh + j), __ldg(xl + j));
    }
    static constexpr int kTile = 2;
    __device__ __forceinline__ const float *gsrc(int i) const { return i == 0 ? xh : xl; }
    __device__ __forceinline__ void add_t(A *a, int k, float v, const float *s, int st, NoSlot) const {
        ds_add_prod(a[k], a[4 + k], v, s[0], s[st]);
    }
    __device__ __forceinline__ Pre pre(const GroupRows &G, int k) const {
        Pre p;
        p.s = (double)s[G.row[k]];
        p.x = x[G.rp[k]];
        return p;
    }
    // the W (hi, lo) partials of row k combined with FP32 two-sums
    template <int W>
    __device__ __forceinline__ static void combine_row(const A (*sh)[NA][32], int lane, int k, A *a) {
        float h = 0.f, l = 0.f;
#pragma unroll
        for (int q = 0; q < W; ++q) {
            const float pp = sh[q][k][lane];
            const float ss = __fadd_rn(h, pp);
            const float bb = __fsub_rn(ss, h);
            l = __fadd_rn(l, __fadd_rn(__fadd_rn(__fsub_rn(h, __fsub_rn(ss, bb)), __fsub_rn(pp, bb)),
                                       sh[q][k + 4][lane]));
            h = ss;
        }
        a[k] = h;
        a[k + 4] = l;
    }
    __device__ __forceinline__ double finish_row(const GroupRows &G, int k, const A *a, const Pre &p) const {
        const double vv = p.s - p.x + ((double)a[k] + (double)a[k + 4]);
        store_h(r, G, k, vv);
        return vv * vv;
    }
};

// x += d, with the double-single split of the new x
template <typename T>
__global__ void k_update_x(int n, const T *__restrict__ d, double *__restrict__ x, float *__restrict__ xh,
                           float *__restrict__ xl) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double v = x[i] + (double)d[i];
    x[i] = v;
    if (xh) {
        float h = (float)v;
        xh[i] = h;
        xl[i] = (float)(v - (double)h);
    }
}

// partial sums of a sweep or residual pass: one per row block (4 per group)
int sweep_blocks(const GridC &g) { return 4 * (g.nz + 1) * g.gpl; }
int resid_blocks(const GridC &g) { return sweep_blocks(g); }

bool stage_fits(int ntmax) { return ntmax > 0; }

// Warps per group (measured on GB300, plume 64 x 64 x 32, interleaved runs):
// the streamed passes run 16 consumer warps per SM; the plain passes with
// programmatic launches are fastest with 6 warps per group while all groups
// fit in one wave of resident blocks, else with the count that fills the
// last wave best.
template <typename T>
int choose_wq_t(const GridC &g) {
    if (sizeof(T) == 4 && g.stage) return 16;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) !=
                                                   cudaSuccess || sms <= 0)
        return 6;
    const long long blocks = (long long)(g.nz + 1) * g.gpl;
    int best = 6;
    double best_eff = -1.0;
    const int cand[3] = {6, 8, 4};
    for (int i = 0; i < 3; ++i) {
        int w = cand[i], bps = 0;
        cudaError_t e;
        if (w == 8)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, k_plain<8, T, OpCheb<T>>, 32 * 8, 0);
        else if (w == 6)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, k_plain<6, T, OpCheb<T>>, 32 * 6, 0);
        else
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, k_plain<4, T, OpCheb<T>>, 32 * 4, 0);
        if (e != cudaSuccess || bps <= 0) continue;
        const double waves = (double)blocks / ((double)sms * bps);
        if (w == 6 && waves <= 1.0) {
            best = 6;
            break;
        }
        const double eff = waves / std::ceil(waves);
        if (eff > best_eff + 1e-9) {
            best_eff = eff;
            best = w;
        }
    }
    cudaGetLastError();  // clear a failed occupancy query
    return best;
}

int choose_wq(const GridC &g, bool fp64) { return fp64 ? choose_wq_t<double>(g) : choose_wq_t<float>(g); }

template <typename T>
void launch_spmv(cudaStream_t st, const GridC &g, const GraphP &gp, const T *val, const T *x, const T *b, T *y) {
    OpSpmv<T, 0> op;
    op.x = x;
    op.b = b;
    op.y = y;
    run_op(st, g, gp, val, op, 0);
}

template <typename T>
void launch_imk(cudaStream_t st, const GridC &g, const GraphP &gp, const T *val, const T *x, T *y) {
    OpSpmv<T, 1> op;
    op.x = x;
    op.b = nullptr;
    op.y = y;
    run_op(st, g, gp, val, op, 0);
}

template <typename T>
void launch_sweep_pow(cudaStream_t st, const GridC &g, const GraphP &gp, const T *val, const T *x, const T *b, T *y,
                      double *part, double *x64, float *xh, float *xl) {
    OpSweepPow<T> op;
    op.x = x;
    op.b = b;
    op.y = y;
    op.part = part;
    op.xu.x = x64;
    op.xu.xh = xh;
    op.xu.xl = xl;
    run_op(st, g, gp, val, op, 0);
}

template <typename T>
void launch_cheb(cudaStream_t st, const GridC &g, const GraphP &gp, const T *val, const T *p, T *r, T *d, T *pn,
                 double c1, double c2, double *x64, float *xh, float *xl) {
    OpCheb<T> op;
    op.xu.x = x64;
    op.xu.xh = xh;
    op.xu.xl = xl;
    op.p = p;
    op.r = r;
    op.d = d;
    op.pn = pn;
    op.c1 = (T)c1;
    op.c2 = (T)c2;
    run_op(st, g, gp, val, op, 0);
}

bool resid_ds_ok(const GridC &g) { return true; }

void launch_resid_ds(cudaStream_t st, const GridC &g, const GraphP &gp, const float *val, const float *s,
                     const double *x, const float *xh, const float *xl, double *r, double *part, int nblk) {
    (void)nblk;
    OpResidDS op;
    op.s = s;
    op.x = x;
    op.xh = xh;
    op.xl = xl;
    op.r = r;
    op.part = part;
    run_op(st, g, gp, val, op, 0);
}

template <typename T>
void launch_update_x(cudaStream_t st, int n, const T *d, double *x, float *xh, float *xl) {
    k_update_x<T><<<(n + 255) / 256, 256, 0, st>>>(n, d, x, xh, xl);
}

template <typename T>
void launch_resid64(cudaStream_t st, const GridC &g, const GraphP &gp, const T *val, const T *s, const double *x,
                    double *r, double *part, int nblk) {
    (void)nblk;
    OpResid64<T> op;
    op.s = s;
    op.x = x;
    op.r = r;
    op.part = part;
    run_op(st, g, gp, val, op, 0);
}


__device__ __forceinline__ double block_sum(double v) {
    __shared__ double red[32];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) red[w] = v;
    __syncthreads();
    double r = 0.0;
    if (threadIdx.x == 0) {
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) r += red[i];
    }
    return r;  // valid in thread 0
}

// ---------------------------------------------------------------------------
// Reductions

// Dot products over the nodes of haloed vectors (each node once, halo
// copies skipped): warp per line of nx nodes, lines strided over the grid.
template <typename A, typename B>
__global__ void k_dots(GridC g, const A *__restrict__ V, size_t ldv, int ncol, const B *__restrict__ y,
                       double *__restrict__ part) {
    const int lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
    const int gw = blockIdx.x * wpb + (threadIdx.x >> 5), nw = gridDim.x * wpb;
    const int nlines = (g.nz + 1) * g.ny;
    for (int k = 0; k < ncol; ++k) {
        const A *v = V + (size_t)k * ldv;
        double acc = 0.0;
        for (int l = gw; l < nlines; l += nw) {
            const int z = l / g.ny, yy = l - z * g.ny;
            const long long base = halo_pos(g, 0, yy, z);
            for (int x = lane; x < g.nx; x += 32) acc += (double)v[base + x] * (double)y[base + x];
        }
        double b = block_sum(acc);
        if (threadIdx.x == 0) part[(size_t)k * gridDim.x + blockIdx.x] = b;
    }
}

// one block per column; fixed strided partial sums then a fixed-order tree
// Column k of the block partials part[k][nblk] summed into out[k] by one
// block of kFinThreads threads: each thread adds its strided share with four
// loads in flight at a time (one memory round trip per four values instead
// of one per value), then the warps' fixed butterflies and warp 0 over the
// warps' sums.  The order depends on nblk only, so the sum is deterministic.
constexpr int kFinThreads = 1024;
__global__ void __launch_bounds__(kFinThreads) k_finalize(const double *__restrict__ part, int nblk, int ncol,
                                                         double *__restrict__ out) {
    __shared__ double sh[32];
    const int k = blockIdx.x;
    const double *p = part + (size_t)k * nblk;
    double s = 0.0;
    int b = threadIdx.x;
    for (; b + 3 * kFinThreads < nblk; b += 4 * kFinThreads) {
        const double a0 = p[b], a1 = p[b + kFinThreads], a2 = p[b + 2 * kFinThreads], a3 = p[b + 3 * kFinThreads];
        s += (a0 + a1) + (a2 + a3);
    }
    for (; b < nblk; b += kFinThreads) s += p[b];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) sh[w] = s;
    __syncthreads();
    if (w == 0) {
        double t = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0.0;
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) out[k] = t;
    }
    (void)ncol;
}

int dot_blocks(const GridC &g) {
    long long b = ((long long)(g.nz + 1) * g.ny + 7) / 8;
    if (b > 296) b = 296;
    if (b < 1) b = 1;
    return (int)b;
}

// The same dot products for FP32 vectors without FP64 arithmetic in the
// pass (FP64 runs at a small fraction of the FP32 rate on this GPU): each
// product and each thread's running sum is kept in FP32-pair arithmetic
// (ds_add_prod, about 48 significant bits), kDotCols columns per pass over
// y; the pairs enter the FP64 block and grid sums only at the end.
constexpr int kDotCols = 8;
// blocks per SM (measured on the 128 x 128 x 40 cloud: 4 beats 2; a flat
// element decomposition at 4 or 8 blocks per SM was slower than warps per line)
constexpr int kDotBlocksPerSM = 4;
// (hi, lo) += (h2, l2) for FP32 pairs, with Knuth's two-sum on the high parts
__device__ __forceinline__ void ds_add_pair(float &hi, float &lo, float h2, float l2) {
    const float s = __fadd_rn(hi, h2);
    const float bb = __fsub_rn(s, hi);
    const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(h2, bb));
    hi = s;
    lo = __fadd_rn(lo, __fadd_rn(err, l2));
}
__global__ void __launch_bounds__(256) k_dots_ds(GridC g, const float *__restrict__ V, size_t ldv, int ncol,
                                                 const float *__restrict__ y, double *__restrict__ part) {
    __shared__ double red[kDotCols][8];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int gw = blockIdx.x * 8 + wid, nw = gridDim.x * 8;
    const int nlines = (g.nz + 1) * g.ny;
    for (int c0 = 0; c0 < ncol; c0 += kDotCols) {
        float hi[kDotCols], lo[kDotCols];
#pragma unroll
        for (int c = 0; c < kDotCols; ++c) hi[c] = lo[c] = 0.f;
        for (int l = gw; l < nlines; l += nw) {
            const int z = l / g.ny, yy = l - z * g.ny;
            const long long base = halo_pos(g, 0, yy, z);
#pragma unroll 4
            for (int x = lane; x < g.nx; x += 32) {
                const float yv = y[base + x];
#pragma unroll
                for (int c = 0; c < kDotCols; ++c)
                    if (c0 + c < ncol) ds_add_prod(hi[c], lo[c], V[(size_t)(c0 + c) * ldv + base + x], yv, 0.f);
            }
        }
        // warp sums in FP32-pair arithmetic; FP64 only for the warps' results
#pragma unroll
        for (int c = 0; c < kDotCols; ++c) {
            float h = hi[c], q = lo[c];
            for (int o = 16; o > 0; o >>= 1)
                ds_add_pair(h, q, __shfl_xor_sync(0xffffffffu, h, o), __shfl_xor_sync(0xffffffffu, q, o));
            if (lane == 0) red[c][wid] = (double)h + (double)q;
        }
        __syncthreads();
        if (threadIdx.x < kDotCols && c0 + (int)threadIdx.x < ncol) {
            double t = 0.0;
            for (int q = 0; q < 8; ++q) t += red[threadIdx.x][q];
            part[(size_t)(c0 + threadIdx.x) * gridDim.x + blockIdx.x] = t;
        }
        __syncthreads();
    }
}

int dot_blocks_ds() {
    static int n = 0;
    if (!n) {
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        n = std::max(1, sms) * kDotBlocksPerSM;
    }
    return n;
}

template <typename A, typename B>
void launch_dots(cudaStream_t st, const GridC &g, const A *V, size_t ldv, int ncol, const B *y, double *part,
                 int nblk, double *out) {
    if constexpr (sizeof(A) == 4 && sizeof(B) == 4) {
        const int nb = std::min(dot_blocks_ds(), std::max(1, (g.nz + 1) * g.ny / 8));
        k_dots_ds<<<nb, 256, 0, st>>>(g, (const float *)V, ldv, ncol, (const float *)y, part);
        k_finalize<<<ncol, kFinThreads, 0, st>>>(part, nb, ncol, out);
        return;
    }
    k_dots<A, B><<<nblk, 256, 0, st>>>(g, V, ldv, ncol, y, part);
    k_finalize<<<ncol, kFinThreads, 0, st>>>(part, nblk, ncol, out);
}

template <typename T>
void launch_sumsq(cudaStream_t st, const GridC &g, const T *x, double *part, int nblk, double *out) {
    launch_dots<T, T>(st, g, x, 0, 1, x, part, nblk, out);
}

// haloed dst <- node-ordered src (every halo copy written)
template <typename T, typename U>
__global__ void k_to_halo(GridC g, const T *__restrict__ src, U *__restrict__ dst) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.n_nodes) return;
    const int z = i / g.nxy, r = i - z * g.nxy, y = r / g.nx, x = r - y * g.nx;
    const long long p = halo_pos(g, x, y, z);
    const int ax = x < g.H ? g.nx : (x >= g.nx - g.H ? -g.nx : 0);
    const int ay = y < g.H ? g.ny * g.nxp : (y >= g.ny - g.H ? -g.ny * g.nxp : 0);
    const U v = (U)src[i];
    dst[p] = v;
    if (ax) dst[p + ax] = v;
    if (ay) {
        dst[p + ay] = v;
        if (ax) dst[p + ax + ay] = v;
    }
}

// node-ordered dst <- haloed src
template <typename U>
__global__ void k_from_halo(GridC g, const U *__restrict__ src, U *__restrict__ dst) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.n_nodes) return;
    const int z = i / g.nxy, r = i - z * g.nxy, y = r / g.nx, x = r - y * g.nx;
    dst[i] = src[halo_pos(g, x, y, z)];
}

template <typename T, typename U>
void launch_to_halo(cudaStream_t st, const GridC &g, const T *src, U *dst) {
    k_to_halo<T, U><<<(g.n_nodes + 255) / 256, 256, 0, st>>>(g, src, dst);
}

template <typename U>
void launch_from_halo(cudaStream_t st, const GridC &g, const U *src, U *dst) {
    k_from_halo<U><<<(g.n_nodes + 255) / 256, 256, 0, st>>>(g, src, dst);
}

void launch_finalize2(cudaStream_t st, const double *part, int nblk, double *out) {
    k_finalize<<<2, kFinThreads, 0, st>>>(part, nblk, 2, out);
}

void launch_finalize(cudaStream_t st, const double *part, int nblk, double *out) {
    k_finalize<<<1, kFinThreads, 0, st>>>(part, nblk, 1, out);
}

// ---------------------------------------------------------------------------
// BiCGStab pass by pass, for scenes too large for the persistent solve.  A
// step is two passes over K (OpBi), each followed by the sums of its dot
// products and one vector kernel; the step's scalars stay on the device
// (every block of the vector kernels forms them from the sums), so a step is
// queued before the host has read back the state of the one before.
// Against GMRES(30) with I + K as preconditioner it needs no basis: on the
// 128 x 128 x 40 cloud an Arnoldi step spent 107 us on orthogonalisation beside
// its two passes of 72 us; a step of this takes 140 us inside a scene's solve, its passes 57 us each with
// what L2 keeps of K (64 with cold caches).
constexpr int kBiParts = 8;  // blocks per sum
template <typename T>
__global__ void __launch_bounds__(512) k_bi_sums(const double *__restrict__ part, size_t stride, int n,
                                                 double *__restrict__ out, const BiState<T> *st) {
    __shared__ double sh[16];
    pdl_trigger();
    pdl_wait();
    if (st->done) return;
    const double *p = part + (size_t)blockIdx.y * stride;
    Dot<T> v;
    const int step = kBiParts * 512;
#pragma unroll 4
    for (int i = blockIdx.x * 512 + threadIdx.x; i < n; i += step) v.join(Dot<T>::from(__ldcg(p + i)));
    v = warp_dot1<T>(v);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v.bits();
    __syncthreads();
    if (threadIdx.x < 32) {
        Dot<T> t;
        if (threadIdx.x < 16) t = Dot<T>::from(sh[threadIdx.x]);
        t = warp_dot1<T>(t);
        if (threadIdx.x == 0) out[blockIdx.y * kBiParts + blockIdx.x] = t.bits();
    }
}
// nd sums of n values, value i of sum w at sums[w * stride + i], by warps
// 0 .. nd - 1, into sh (synchronises)
template <typename T>
__device__ __forceinline__ void bi_total(const double *sums, size_t stride, int n, int nd, double *sh) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (w < nd) {
        Dot<T> v;
        for (int i = lane; i < n; i += 32) v.join(Dot<T>::from(__ldcg(sums + w * stride + i)));
        v = warp_dot1<T>(v);
        if (lane == 0) sh[w] = v.bits();
    }
    __syncthreads();
}
// b = r64 scaled by a power of two; r = p = b, d = 0; the state of a new solve
template <typename T>
__global__ void k_bi_start(int n, const double *__restrict__ r64, T down, T bb, T stop2, T *__restrict__ b,
                           T *__restrict__ r, T *__restrict__ p, T *__restrict__ d, BiState<T> *st) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) {
        BiState<T> s{};
        s.rho = s.best = s.rn = bb;
        s.stop2 = stop2;
        *st = s;
    }
    if (i >= n) return;
    const T v = down * (T)r64[i];
    b[i] = v;
    r[i] = v;
    p[i] = v;
    d[i] = T(0);
}
// The vector kernels: four elements per thread in 16-byte accesses, the first
// four loaded before the sums are formed, so that the two latencies overlap
// (vectors in L2; 2.4 us less per step of the 128 x 128 x 40 cloud, whose run
// takes 19.8 ms instead of 20.2 with one element at a time).
template <typename T>
struct alignas(16) Quad {
    T v[4];
};
// alpha = rho / r0.v; d += alpha p; r <- s = r - alpha v
template <typename T>
__global__ void __launch_bounds__(256) k_bi_s(int n, const double *__restrict__ sums, size_t stride, int ns,
                                              const T *__restrict__ p, const T *__restrict__ v, T *__restrict__ r,
                                              T *__restrict__ d, BiState<T> *st) {
    __shared__ double sh[8];
    __shared__ T sa;
    pdl_trigger();
    pdl_wait();
    if (st->done) return;
    using Q = Quad<T>;
    const int n4 = n / 4, step = gridDim.x * blockDim.x;
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    Q pq, vq, rq, dq;
    auto load = [&]() {
        pq = reinterpret_cast<const Q *>(p)[i];
        vq = reinterpret_cast<const Q *>(v)[i];
        rq = reinterpret_cast<Q *>(r)[i];
        dq = reinterpret_cast<Q *>(d)[i];
    };
    if (i < n4) load();
    bi_total<T>(sums, stride, ns, 1, sh);
    if (threadIdx.x == 0) {
        const T r0v = Dot<T>::from(sh[0]).value();
        sa = r0v != T(0) ? st->rho / r0v : T(0);
        if (blockIdx.x == 0) st->alpha = sa;
    }
    __syncthreads();
    const T a = sa;
    while (i < n4) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            dq.v[k] += a * pq.v[k];
            rq.v[k] -= a * vq.v[k];
        }
        reinterpret_cast<Q *>(d)[i] = dq;
        reinterpret_cast<Q *>(r)[i] = rq;
        i += step;
        if (i < n4) load();
    }
    const int e = 4 * n4 + threadIdx.x;  // up to three more
    if (blockIdx.x == 0 && e < n) {
        d[e] += a * p[e];
        r[e] -= a * v[e];
    }
}
// omega, beta and the new rho from the sums; d += omega s; r = s - omega t;
// p = r + beta (p - omega v).  The last block to finish writes the state,
// which the others read.
template <typename T>
__global__ void __launch_bounds__(256) k_bi_p(int n, const double *__restrict__ sums, size_t stride, int ns,
                                              const T *__restrict__ v,
                                              const T *__restrict__ t, T *__restrict__ r, T *__restrict__ p,
                                              T *__restrict__ d, BiState<T> *st) {
    __shared__ double sh[8];
    __shared__ T sv[4];
    pdl_trigger();
    pdl_wait();
    if (st->done) return;
    using Q = Quad<T>;
    const int n4 = n / 4, step = gridDim.x * blockDim.x;
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    Q rq, tq, pq, vq, dq;
    auto load = [&]() {
        rq = reinterpret_cast<Q *>(r)[i];
        tq = reinterpret_cast<const Q *>(t)[i];
        pq = reinterpret_cast<Q *>(p)[i];
        vq = reinterpret_cast<const Q *>(v)[i];
        dq = reinterpret_cast<Q *>(d)[i];
    };
    if (i < n4) load();
    bi_total<T>(sums, stride, ns, 5, sh);
    if (threadIdx.x == 0) {
        const Dot<T> ts = Dot<T>::from(sh[0]), tt = Dot<T>::from(sh[1]), r0t = Dot<T>::from(sh[3]);
        Dot<T> r0r = Dot<T>::from(sh[2]), rn = Dot<T>::from(sh[4]);
        const T om = tt.value() > T(0) ? ts.value() / tt.value() : T(0);
        r0t.add_to(r0r, -om);       // r0.r = r0.s - omega r0.t
        ts.add_to(rn, T(-2) * om);  // r.r = s.s - 2 omega t.s + omega^2 t.t
        Dot<T> ott;
        tt.add_to(ott, om);
        ott.add_to(rn, om);
        sv[0] = om;
        sv[2] = r0r.value();
        sv[3] = rn.value();
        const T rho = st->rho;
        sv[1] = (rho != T(0) && om != T(0)) ? (sv[2] / rho) * (st->alpha / om) : T(0);
    }
    __syncthreads();
    const T om = sv[0], be = sv[1];
    auto one = [&](T &rv, T tv, T &pv, T vv, T &dv) {
        const T s = rv, rr = s - om * tv;
        dv += om * s;
        pv = rr + be * (pv - om * vv);
        rv = rr;
    };
    while (i < n4) {
#pragma unroll
        for (int k = 0; k < 4; ++k) one(rq.v[k], tq.v[k], pq.v[k], vq.v[k], dq.v[k]);
        reinterpret_cast<Q *>(d)[i] = dq;
        reinterpret_cast<Q *>(p)[i] = pq;
        reinterpret_cast<Q *>(r)[i] = rq;
        i += step;
        if (i < n4) load();
    }
    const int e = 4 * n4 + threadIdx.x;  // up to three more
    if (blockIdx.x == 0 && e < n) one(r[e], t[e], p[e], v[e], d[e]);
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&st->left, 1u) + 1u == gridDim.x) {  // every block has read the old state
            st->left = 0;
            st->rho = sv[2];
            st->rn = sv[3];
            st->steps += 1;
            if (sv[3] < st->best) {
                st->best = sv[3];
                st->since = 0;
            } else {
                st->since += 1;
            }
            if (!(sv[3] > st->stop2) || om == T(0) || !(fabs(be) > T(0)) || st->since > 40) st->done = 1;
        }
    }
}
// x += up * d, with the FP32 pair of the new x
template <typename T>
__global__ void k_bi_end(int n, const T *__restrict__ d, T up, double *__restrict__ x, float *__restrict__ xh,
                         float *__restrict__ xl) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double v = x[i] + (double)(up * d[i]);
    x[i] = v;
    if (xh) {
        const float h = (float)v;
        xh[i] = h;
        xl[i] = (float)(v - (double)h);
    }
}

size_t bi_part_words(const GridC &g) { return (size_t)5 * sweep_blocks(g) + 8 * kBiParts; }

template <typename T>
void launch_bi_start(cudaStream_t st, int n, const double *r64, double down, double bb, double stop2, T *b, T *r,
                     T *p, T *d, BiState<T> *state) {
    k_bi_start<T><<<(n + 255) / 256, 256, 0, st>>>(n, r64, (T)down, (T)bb, (T)stop2, b, r, p, d, state);
}
template <typename T>
void launch_bi_step(cudaStream_t st, const GridC &g, const GraphP &gp, const T *val, const T *r0, T *r, T *p, T *v,
                    T *t, T *d, double *part, BiState<T> *state, long long *launches) {
    const int n = (int)g.npad, np = sweep_blocks(g);
    double *sums = part + (size_t)5 * np;
    int dev = 0, nsm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || nsm < 1)
        nsm = 152;
    const int nb = std::max(1, std::min((n / 4 + 255) / 256, 8 * nsm));  // at most 8 blocks per SM
    auto go = [&](auto kern, dim3 blocks, int threads, auto... args) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = blocks;
        cfg.blockDim = dim3(threads);
        cfg.stream = st;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        cudaLaunchKernelEx(&cfg, kern, args...);
    };
    const double *cpart = part, *csums = sums;
    const T *cp = p, *cv = v, *ct = t;
    const BiState<T> *cst = state;
    OpBi<T, 1> ov{p, r0, v, part, (size_t)np, state};
    OpBi<T, 5> ot{r, r0, t, part, (size_t)np, state};
    // passes in rounds leave a value per block, which the vector kernels sum
    // themselves (two launches less per step: 10 us of 152 on the cloud)
    bool rounds = false;
    if constexpr (sizeof(T) == 4) rounds = run_in_rounds<OpBi<T, 1>>(g, gp) && run_in_rounds<OpBi<T, 5>>(g, gp);
    const size_t stride = rounds ? (size_t)np : kBiParts;
    const int ns = rounds ? gp.rd_nb : kBiParts;
    if (rounds) csums = part;
    run_op(st, g, gp, val, ov, 0);
    if (!rounds) go(k_bi_sums<T>, dim3(kBiParts, 1), 512, cpart, (size_t)np, np, sums, cst);
    go(k_bi_s<T>, dim3(nb), 256, n, csums, stride, ns, cp, cv, r, d, state);
    run_op(st, g, gp, val, ot, 0);
    if (!rounds) go(k_bi_sums<T>, dim3(kBiParts, 5), 512, cpart, (size_t)np, np, sums, cst);
    go(k_bi_p<T>, dim3(nb), 256, n, csums, stride, ns, cv, ct, r, p, d, state);
    *launches += rounds ? 4 : 6;
}
template <typename T>
void launch_bi_end(cudaStream_t st, int n, const T *d, double up, double *x, float *xh, float *xl) {
    k_bi_end<T><<<(n + 255) / 256, 256, 0, st>>>(n, d, (T)up, x, xh, xl);
}

// ---------------------------------------------------------------------------
// Vector operations

template <typename T, typename U>
__global__ void k_convert(int n, const T *__restrict__ a, U *__restrict__ b) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) b[i] = (U)a[i];
}
template <typename T>
__global__ void k_axpy64(int n, const T *__restrict__ d, double *__restrict__ x) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) x[i] += (double)d[i];
}
template <typename T>
__global__ void k_scale(int n, const T *__restrict__ a, double alpha, T *__restrict__ b) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) b[i] = (T)(alpha * (double)a[i]);
}
template <typename T>
__global__ void k_add(int n, T *a, const T *b) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) a[i] += b[i];
}
template <typename T>
__global__ void k_cheb_start(int n, const double *__restrict__ r64, double alpha, T *__restrict__ b,
                             T *__restrict__ d, T *__restrict__ p) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const T v = (T)r64[i];
    b[i] = v;
    d[i] = T(0);
    p[i] = (T)(alpha * (double)v);
}
template <typename T>
__global__ void k_gupdate(int n, T *__restrict__ w, const T *__restrict__ V, size_t ldv, int k,
                          const double *__restrict__ h, double sign) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double acc = (double)w[i];
    for (int j = 0; j < k; ++j) acc += sign * h[j] * (double)V[(size_t)j * ldv + i];
    w[i] = (T)acc;
}

// w += sign sum_j h_j V_j for FP32 vectors in FP32-pair arithmetic: the
// coefficients are split once per block into (high, low) FP32 pairs, and
// each element's sum is carried as a pair and rounded to FP32 at the end
constexpr int kGupdateMaxK = 64;
template <bool kNorm>
__global__ void __launch_bounds__(256) k_gupdate_ds(GridC g, int n, float *__restrict__ w, const float *__restrict__ V,
                                                    size_t ldv, int k, const double *__restrict__ h, double sign,
                                                    double *__restrict__ part) {
    __shared__ float hh[kGupdateMaxK], hl[kGupdateMaxK];
    __shared__ double red[8];
    for (int j = threadIdx.x; j < k; j += blockDim.x) {
        const double c = sign * h[j];
        const float a = (float)c;
        hh[j] = a;
        hl[j] = (float)(c - (double)a);
    }
    __syncthreads();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    float r = 0.f;
    if (i < n) {
        float hi = w[i], lo = 0.f;
#pragma unroll 4
        for (int j = 0; j < k; ++j) ds_add_prod(hi, lo, V[(size_t)j * ldv + i], hh[j], hl[j]);
        r = __fadd_rn(hi, lo);
        w[i] = r;
    }
    if constexpr (kNorm) {
        // ||w||^2 over the interior (halo copies excluded), as FP32 pairs per
        // warp and FP64 per block: part[blockIdx.x]
        float sh = 0.f, sl = 0.f;
        if (i < n) {
            const int rem = i % g.lp, yy = rem / g.nxp, xx = rem - yy * g.nxp;
            if (xx >= g.H && xx < g.nx + g.H && yy >= g.H && yy < g.ny + g.H) ds_add_prod(sh, sl, r, r, 0.f);
        }
        for (int o = 16; o > 0; o >>= 1)
            ds_add_pair(sh, sl, __shfl_xor_sync(0xffffffffu, sh, o), __shfl_xor_sync(0xffffffffu, sl, o));
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = (double)sh + (double)sl;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            for (int q = 0; q < (int)(blockDim.x >> 5); ++q) t += red[q];
            part[blockIdx.x] = t;
        }
    }
}

template <typename T, typename U>
void launch_convert(cudaStream_t st, int n, const T *a, U *b) {
    k_convert<T, U><<<(n + 255) / 256, 256, 0, st>>>(n, a, b);
}
template <typename T>
void launch_axpy_to64(cudaStream_t st, int n, const T *d, double *x) {
    k_axpy64<T><<<(n + 255) / 256, 256, 0, st>>>(n, d, x);
}
template <typename T>
void launch_scale(cudaStream_t st, int n, const T *a, double alpha, T *b) {
    k_scale<T><<<(n + 255) / 256, 256, 0, st>>>(n, a, alpha, b);
}
template <typename T>
void launch_add(cudaStream_t st, int n, T *a, const T *b) {
    k_add<T><<<(n + 255) / 256, 256, 0, st>>>(n, a, b);
}
template <typename T>
void launch_cheb_start(cudaStream_t st, int n, const double *r64, double alpha, T *b, T *d, T *p) {
    k_cheb_start<T><<<(n + 255) / 256, 256, 0, st>>>(n, r64, alpha, b, d, p);
}
template <typename T>
void launch_gmres_update(cudaStream_t st, int n, T *w, const T *V, size_t ldv, int k, const double *h) {
    if constexpr (sizeof(T) == 4) {
        k_gupdate_ds<false><<<(n + 255) / 256, 256, 0, st>>>(GridC(), n, (float *)w, (const float *)V, ldv, k, h,
                                                               -1.0, nullptr);
        return;
    }
    k_gupdate<T><<<(n + 255) / 256, 256, 0, st>>>(n, w, V, ldv, k, h, -1.0);
}
// w -= V h, then ||w||^2 (interior) into *out; part: scratch partial sums
template <typename T>
void launch_gmres_update_norm(cudaStream_t st, const GridC &g, int n, T *w, const T *V, size_t ldv, int k,
                              const double *h, double *part, int nblk, double *out) {
    if constexpr (sizeof(T) == 4) {
        const int nb = (n + 255) / 256;
        k_gupdate_ds<true><<<nb, 256, 0, st>>>(g, n, (float *)w, (const float *)V, ldv, k, h, -1.0, part);
        k_finalize<<<1, kFinThreads, 0, st>>>(part, nb, 1, out);
        return;
    }
    launch_gmres_update<T>(st, n, w, V, ldv, k, h);
    launch_sumsq<T>(st, g, w, part, nblk, out);
}

template <typename T>
void launch_combine(cudaStream_t st, int n, T *x, const T *V, size_t ldv, int k, const double *y) {
    if constexpr (sizeof(T) == 4) {
        k_gupdate_ds<false><<<(n + 255) / 256, 256, 0, st>>>(GridC(), n, (float *)x, (const float *)V, ldv, k, y, 1.0,
                                                               nullptr);
        return;
    }
    k_gupdate<T><<<(n + 255) / 256, 256, 0, st>>>(n, x, V, ldv, k, y, 1.0);
}

template <typename T>
__global__ void k_axpby(int n, double a, const T *__restrict__ x, double b, const T *__restrict__ y,
                        T *__restrict__ out) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = (T)(a * (double)x[i] + b * (double)y[i]);
}
template <typename T>
void launch_axpby(cudaStream_t st, int n, double a, const T *x, double b, const T *y, T *out) {
    k_axpby<T><<<(n + 255) / 256, 256, 0, st>>>(n, a, x, b, y, out);
}

#define BINST(T)                                                                                                   \
    template void launch_bi_start<T>(cudaStream_t, int, const double *, double, double, double, T *, T *, T *, T *, \
                                     BiState<T> *);                                                                \
    template void launch_bi_step<T>(cudaStream_t, const GridC &, const GraphP &, const T *, const T *, T *, T *,   \
                                    T *, T *, T *, double *, BiState<T> *, long long *);                           \
    template void launch_bi_end<T>(cudaStream_t, int, const T *, double, double *, float *, float *);
BINST(float)
BINST(double)
#undef BINST

#define INST(T)                                                                                                    \
    template void launch_spmv<T>(cudaStream_t, const GridC &, const GraphP &, const T *, const T *, const T *, T *); \
    template void launch_imk<T>(cudaStream_t, const GridC &, const GraphP &, const T *, const T *, T *);             \
    template void launch_resid64<T>(cudaStream_t, const GridC &, const GraphP &, const T *, const T *,               \
                                    const double *, double *, double *, int);                                       \
    template void launch_dots<T, T>(cudaStream_t, const GridC &, const T *, size_t, int, const T *, double *, int,  \
                                    double *);                                                                      \
    template void launch_sumsq<T>(cudaStream_t, const GridC &, const T *, double *, int, double *);                 \
    template void launch_to_halo<T, double>(cudaStream_t, const GridC &, const T *, double *);                      \
    template void launch_from_halo<T>(cudaStream_t, const GridC &, const T *, T *);                                 \
    template void launch_axpy_to64<T>(cudaStream_t, int, const T *, double *);                                      \
    template void launch_scale<T>(cudaStream_t, int, const T *, double, T *);                                       \
    template void launch_cheb_start<T>(cudaStream_t, int, const double *, double, T *, T *, T *);                  \
    template void launch_add<T>(cudaStream_t, int, T *, const T *);                                                \
    template void launch_gmres_update<T>(cudaStream_t, int, T *, const T *, size_t, int, const double *);           \
    template void launch_gmres_update_norm<T>(cudaStream_t, const GridC &, int, T *, const T *, size_t, int,       \
                                              const double *, double *, int, double *);                          \
    template void launch_combine<T>(cudaStream_t, int, T *, const T *, size_t, int, const double *);            \
    template void launch_axpby<T>(cudaStream_t, int, double, const T *, double, const T *, T *);                   \
    template void launch_update_x<T>(cudaStream_t, int, const T *, double *, float *, float *);                   \
    template void launch_sweep_pow<T>(cudaStream_t, const GridC &, const GraphP &, const T *, const T *,          \
                                      const T *, T *, double *, double *, float *, float *);                    \
    template void launch_cheb<T>(cudaStream_t, const GridC &, const GraphP &, const T *, const T *, T *, T *,     \
                                 T *, double, double, double *, float *, float *);
INST(float)
INST(double)
#undef INST
template void launch_to_halo<float, float>(cudaStream_t, const GridC &, const float *, float *);
template void launch_convert<double, float>(cudaStream_t, int, const double *, float *);
template void launch_convert<float, double>(cudaStream_t, int, const float *, double *);
template void launch_convert<double, double>(cudaStream_t, int, const double *, double *);
template void launch_convert<float, float>(cudaStream_t, int, const float *, float *);

}  // namespace tk
