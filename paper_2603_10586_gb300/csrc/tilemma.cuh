// Register-tile products on operands staged in shared memory: a warp holds 16 RA
// rows x 2 J columns, RA x J complex accumulators per thread (thread tr = lane
// & 15 takes rows tr + 16 i, or two neighbouring rows at a time; tc = lane >> 4
// takes columns tc + 2 j).
#pragma once
#include <type_traits>

#include "farmac.cuh"

namespace vie {

__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool valid) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    const int n = valid ? 16 : 0;  // 0 source bytes: zero fill
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// columns per thread of a full warp tile (two threads side by side): float32
// wants few shared-memory loads per FMA, float64 is bound by its units, and
// double-float (44 float32 operations per product) wants registers for more warps
template <class TX> constexpr int kJ = 8;
template <> constexpr int kJ<double2> = 4;
template <> constexpr int kJ<float4> = 2;

// elements per 16-byte copy or shared-memory load
template <class T> constexpr int kE = 16 / (int)sizeof(T);

template <class TA, int RA, int J> __device__ __forceinline__ void zero_acc(TA (&acc)[RA][J]) {
#pragma unroll
    for (int i = 0; i < RA; ++i)
#pragma unroll
        for (int j = 0; j < J; ++j) acc[i][j] = acc_zero<TA>();
}

// float32: packed FMAs, (re, im) += a.re (b.re, b.im) + a.im (-b.im, b.re)
// (conj: + a.im (b.im, -b.re)), the products and their order as in mac / mac_conj;
// two lanes' worth per instruction leaves issue slots for the loads
__device__ __forceinline__ unsigned long long pack2(float x, float y) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ void fma2(float2& acc, unsigned long long a, unsigned long long b) {
    unsigned long long c = pack2(acc.x, acc.y);
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(acc.x), "=f"(acc.y) : "l"(c));
}

// one 16-byte unit of shared memory: two float32 values or one wider one
__device__ __forceinline__ void ld16(float2 (&v)[2], const float2* p) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    v[0] = make_float2(q.x, q.y);
    v[1] = make_float2(q.z, q.w);
}
__device__ __forceinline__ void ld16(float4 (&v)[1], const float4* p) { v[0] = *p; }
__device__ __forceinline__ void ld16(double2 (&v)[1], const double2* p) { v[0] = *p; }

template <class TF, class TX, class TA, int RA, int J, bool CONJ>
__device__ __forceinline__ void outer(TA (&acc)[RA][J], const TF (&av)[RA], const TX (&bv)[J]) {
    if constexpr (std::is_same<TA, float2>::value) {
        unsigned long long ar[RA], ai[RA];
#pragma unroll
        for (int i = 0; i < RA; ++i) {
            ar[i] = pack2(av[i].x, av[i].x);
            ai[i] = pack2(av[i].y, av[i].y);
        }
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const unsigned long long b = pack2(bv[j].x, bv[j].y);
            const unsigned long long r = CONJ ? pack2(bv[j].y, -bv[j].x) : pack2(-bv[j].y, bv[j].x);
#pragma unroll
            for (int i = 0; i < RA; ++i) {
                fma2(acc[i][j], ar[i], b);
                fma2(acc[i][j], ai[i], r);
            }
        }
    } else {
#pragma unroll
        for (int i = 0; i < RA; ++i)
#pragma unroll
            for (int j = 0; j < J; ++j) {
                if (CONJ) mac_conj(acc[i][j], av[i], bv[j]);
                else mac(acc[i][j], av[i], bv[j]);
            }
    }
}

// acc += A B over KG K values, A [row][K] (phase 1) or [K][row] (phase 2); A, B at
// the thread's first row and column
template <class TF, class TX, class TA, int PHASE, int KG, int LA, int LB, int RA, int J>
__device__ __forceinline__ void mma_stage(const TF* A, const TX* B, TA (&acc)[RA][J]) {
    constexpr int EA = kE<TF>, EB = kE<TX>, KS = EA > EB ? EA : EB;  // K values per step
#pragma unroll 1
    for (int k = 0; k < KG; k += KS) {
        TF av[KS][RA];
        TX bv[KS][J];
        if constexpr (PHASE == 1) {
#pragma unroll
            for (int i = 0; i < RA; ++i)
#pragma unroll
                for (int e = 0; e < KS; e += EA) {
                    TF v[EA];
                    ld16(v, A + 16 * i * LA + k + e);
#pragma unroll
                    for (int f = 0; f < EA; ++f) av[e + f][i] = v[f];
                }
        } else {
#pragma unroll
            for (int e = 0; e < KS; ++e)
#pragma unroll
                for (int i = 0; i < RA; i += EA) {
                    TF v[EA];
                    ld16(v, A + (k + e) * LA + 16 * i);
#pragma unroll
                    for (int f = 0; f < EA; ++f) av[e][i + f] = v[f];
                }
        }
#pragma unroll
        for (int j = 0; j < J; ++j)
#pragma unroll
            for (int e = 0; e < KS; e += EB) {
                TX v[EB];
                ld16(v, B + 2 * j * LB + k + e);
#pragma unroll
                for (int f = 0; f < EB; ++f) bv[e + f][j] = v[f];
            }
#pragma unroll
        for (int e = 0; e < KS; ++e) outer<TF, TX, TA, RA, J, PHASE == 1>(acc, av[e], bv[e]);
    }
}

}  // namespace vie
