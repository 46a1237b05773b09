// Multiply-accumulate and stores of the far-apply kernels in the three
// arithmetics they share: complex float32, complex float64 and double-float
// (float4 vectors) with complex float32 factors.
#pragma once
#include "cplx.cuh"

namespace vie {

template <class T2> __device__ __forceinline__ T2 shfl_down2(T2 v, int o) {
    v.x = __shfl_down_sync(0xffffffffu, v.x, o);
    v.y = __shfl_down_sync(0xffffffffu, v.y, o);
    return v;
}

// ---------------------------------------------------------------------------
// Accumulation.  Float32 and float64 vectors accumulate in their own
// precision.  For the float64 refinement residual the vectors come split into
// float32 head + tail (float4: re_h, im_h, re_l, im_l) and the products with
// the exact float32 factors are summed in double-float arithmetic: each
// product is formed exactly with an FMA (Dekker's two-product), each addition
// keeps its rounding error (Knuth's two-sum), so a sum carries about 48
// significant bits while every operation runs on the float32 pipes (the
// float64 pipe of this GPU is a small fraction of the float32 one).
// ---------------------------------------------------------------------------
struct Dfc { float rh, rl, ih, il; };  // (rh + rl) + j (ih + il)

template <class TX> struct AccOf { using t = TX; };
template <> struct AccOf<float4> { using t = Dfc; };

template <class TA> __device__ __forceinline__ TA acc_zero();
template <> __device__ __forceinline__ float2 acc_zero<float2>() { return make_float2(0.f, 0.f); }
template <> __device__ __forceinline__ double2 acc_zero<double2>() { return make_double2(0.0, 0.0); }
template <> __device__ __forceinline__ Dfc acc_zero<Dfc>() { return {0.f, 0.f, 0.f, 0.f}; }

// acc += conj(a) x  and  acc += a x
__device__ __forceinline__ void mac_conj(float2& acc, float2 a, float2 x) { cfmac(acc, a, x); }
__device__ __forceinline__ void mac_conj(double2& acc, float2 a, double2 x) { cfmac(acc, cvt<double2>(a), x); }
__device__ __forceinline__ void mac_conj(double2& acc, double2 a, double2 x) { cfmac(acc, a, x); }
__device__ __forceinline__ void mac(float2& acc, float2 a, float2 x) { cfma(acc, a, x); }
__device__ __forceinline__ void mac(double2& acc, float2 a, double2 x) { cfma(acc, cvt<double2>(a), x); }
__device__ __forceinline__ void mac(double2& acc, double2 a, double2 x) { cfma(acc, a, x); }

// (h, l) += a (bh + bl): the product a bh exactly as p + e, the tail a bl
// folded into e, then h + p by two-sum with its error and e added to l.
// The _rn intrinsics keep the compiler from fusing these steps.
__device__ __forceinline__ void df_acc(float& h, float& l, float a, float bh, float bl) {
    const float p = __fmul_rn(a, bh);
    float e = fmaf(a, bh, -p);
    e = fmaf(a, bl, e);
    const float sum = __fadd_rn(h, p);
    const float bv = __fsub_rn(sum, h);
    const float err = __fadd_rn(__fsub_rn(h, __fsub_rn(sum, bv)), __fsub_rn(p, bv));
    h = sum;
    l = __fadd_rn(l, __fadd_rn(err, e));
}
__device__ __forceinline__ void mac_conj(Dfc& acc, float2 a, float4 x) {
    df_acc(acc.rh, acc.rl, a.x, x.x, x.z);
    df_acc(acc.rh, acc.rl, a.y, x.y, x.w);
    df_acc(acc.ih, acc.il, a.x, x.y, x.w);
    df_acc(acc.ih, acc.il, -a.y, x.x, x.z);
}
__device__ __forceinline__ void mac(Dfc& acc, float2 a, float4 x) {
    df_acc(acc.rh, acc.rl, a.x, x.x, x.z);
    df_acc(acc.rh, acc.rl, -a.y, x.y, x.w);
    df_acc(acc.ih, acc.il, a.x, x.y, x.w);
    df_acc(acc.ih, acc.il, a.y, x.x, x.z);
}

__device__ __forceinline__ void acc_add(float2& a, float2 b) { a += b; }
__device__ __forceinline__ void acc_add(double2& a, double2 b) { a += b; }
__device__ __forceinline__ void df_add(float& h, float& l, float bh, float bl) {
    const float sum = __fadd_rn(h, bh);
    const float bv = __fsub_rn(sum, h);
    const float err = __fadd_rn(__fsub_rn(h, __fsub_rn(sum, bv)), __fsub_rn(bh, bv));
    h = sum;
    l = __fadd_rn(__fadd_rn(l, bl), err);
}
__device__ __forceinline__ void acc_add(Dfc& a, const Dfc& b) {
    df_add(a.rh, a.rl, b.rh, b.rl);
    df_add(a.ih, a.il, b.ih, b.il);
}

__device__ __forceinline__ float2 acc_shfl_down(float2 v, int o) { return shfl_down2(v, o); }
__device__ __forceinline__ double2 acc_shfl_down(double2 v, int o) { return shfl_down2(v, o); }
__device__ __forceinline__ Dfc acc_shfl_down(Dfc v, int o) {
    return {__shfl_down_sync(0xffffffffu, v.rh, o), __shfl_down_sync(0xffffffffu, v.rl, o),
            __shfl_down_sync(0xffffffffu, v.ih, o), __shfl_down_sync(0xffffffffu, v.il, o)};
}

__device__ __forceinline__ void store(float2* p, float2 v) { *p = v; }
__device__ __forceinline__ void store(double2* p, double2 v) { *p = v; }
__device__ __forceinline__ void store(double2* p, const Dfc& v) {
    *p = make_double2((double)v.rh + (double)v.rl, (double)v.ih + (double)v.il);
}
// renormalised head + tail (fast two-sum, the head dominates)
__device__ __forceinline__ void store(float4* p, const Dfc& v) {
    const float sr = __fadd_rn(v.rh, v.rl), si = __fadd_rn(v.ih, v.il);
    *p = make_float4(sr, si, __fsub_rn(v.rl, __fsub_rn(sr, v.rh)), __fsub_rn(v.il, __fsub_rn(si, v.ih)));
}

// a stored vector element as an accumulator
__device__ __forceinline__ float2 as_acc(float2 v) { return v; }
__device__ __forceinline__ double2 as_acc(double2 v) { return v; }
__device__ __forceinline__ Dfc as_acc(float4 v) { return {v.x, v.z, v.y, v.w}; }

}  // namespace vie
