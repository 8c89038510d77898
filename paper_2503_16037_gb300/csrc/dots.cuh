// Dot products of the BiCGStab solves.
#pragma once
#include <cuda_runtime.h>

namespace tk {

// Sums of products: FP32 pairs (exact products, compensated sums, about 48
// bits) for FP32 scenes, FP64 otherwise.  bits() / from() carry one through an
// 8-byte word.
template <typename T>
struct Dot;
template <>
struct Dot<float> {
    float h = 0.f, l = 0.f;
    __device__ __forceinline__ void add(float a, float b) {
        const float p = __fmul_rn(a, b);
        add2(p, fmaf(a, b, -p));
    }
    __device__ __forceinline__ void add2(float p, float e) {
        const float s = __fadd_rn(h, p);
        const float bb = __fsub_rn(s, h);
        const float err = __fadd_rn(__fsub_rn(h, __fsub_rn(s, bb)), __fsub_rn(p, bb));
        h = s;
        l = __fadd_rn(l, __fadd_rn(err, e));
    }
    __device__ __forceinline__ Dot xch(int o) const {
        Dot r;
        r.h = __shfl_xor_sync(0xffffffffu, h, o);
        r.l = __shfl_xor_sync(0xffffffffu, l, o);
        return r;
    }
    __device__ __forceinline__ void join(const Dot &q) { add2(q.h, q.l); }
    // c * (this) added to d, c exact
    __device__ __forceinline__ void add_to(Dot &d, float c) const {
        d.add(c, h);
        d.l = fmaf(c, l, d.l);
    }
    __device__ __forceinline__ float value() const { return h + l; }
    __device__ __forceinline__ double bits() const {
        return __hiloint2double(__float_as_int(h), __float_as_int(l));
    }
    __device__ __forceinline__ static Dot from(double b) {
        Dot d;
        d.h = __int_as_float(__double2hiint(b));
        d.l = __int_as_float(__double2loint(b));
        return d;
    }
};
template <>
struct Dot<double> {
    double h = 0.0;
    __device__ __forceinline__ void add(double a, double b) { h = fma(a, b, h); }
    __device__ __forceinline__ Dot xch(int o) const {
        Dot r;
        r.h = __shfl_xor_sync(0xffffffffu, h, o);
        return r;
    }
    __device__ __forceinline__ void join(const Dot &q) { h += q.h; }
    __device__ __forceinline__ void add_to(Dot &d, double c) const { d.h = fma(c, h, d.h); }
    __device__ __forceinline__ double value() const { return h; }
    __device__ __forceinline__ double bits() const { return h; }
    __device__ __forceinline__ static Dot from(double b) {
        Dot d;
        d.h = b;
        return d;
    }
};

// N = 8 sums over the warp in 9 joins: the lanes split the sums between
// them stage by stage; lane i ends with sum number (i >> 2)
template <typename T>
__device__ __forceinline__ Dot<T> warp_dots8(Dot<T> (&v)[8]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int st = 4; st >= 1; st >>= 1) {
        const int o = 4 * st;  // 16, 8, 4
        const bool hi = lane & o;
#pragma unroll
        for (int i = 0; i < st; ++i) {
            const Dot<T> give = hi ? v[i] : v[i + st];
            Dot<T> keep = hi ? v[i + st] : v[i];
            keep.join(give.xch(o));
            v[i] = keep;
        }
    }
    v[0].join(v[0].xch(2));
    v[0].join(v[0].xch(1));
    return v[0];
}
template <typename T>
__device__ __forceinline__ Dot<T> warp_dot1(Dot<T> v) {
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) v.join(v.xch(o));
    return v;
}

}  // namespace tk
