// tcgen05 / mbarrier / tensor-memory helpers and the bf16 operand split shared by
// the tensor-core far applies (apply_umma.cu, apply_ws.cu).
#pragma once
#include <cuda_bf16.h>

#include <cstdint>

namespace vie {

constexpr long long kWaitCycles = 2000000000LL;  // ~1 s at 2 GHz

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// shared-memory matrix descriptor, canonical layout without swizzle: 8 x 8 core
// matrices of 128 contiguous bytes, `lbo` bytes apart along K, `sbo` between
// 8-row groups
__device__ __forceinline__ uint64_t sdesc(uint32_t addr, uint32_t lbo, uint32_t sbo = 128) {
    uint64_t d = (uint64_t)((addr >> 4) & 0x3FFFu);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;  // descriptor version of this architecture
    return d;                // base offset 0, relative LBO, no swizzle
}

// instruction descriptor of kind::f16: bf16 x bf16 -> f32, both K-major,
// M = 128, N = n
__host__ __device__ constexpr uint32_t idesc(int n, bool neg_a) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (neg_a ? (1u << 13) : 0u) | ((uint32_t)(n >> 3) << 17) |
           (8u << 24);
}

__device__ __forceinline__ void umma(uint32_t dt, uint64_t ad, uint64_t bd, uint32_t id, uint32_t acc) {
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(dt),
        "l"(ad), "l"(bd), "r"(id), "r"(acc));
}

__device__ __forceinline__ void umma_commit(uint32_t mbar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar)
                 : "memory");
}

__device__ __forceinline__ void mbar_init(uint32_t mbar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mbar) : "memory");
}

// bounded wait for the completion of the phase with the given parity
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity) {
    const long long t0 = clock64();
    while (true) {
        uint32_t ok;
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(mbar), "r"(parity)
            : "memory");
        if (ok) return true;
        if (clock64() - t0 > kWaitCycles) return false;
    }
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// split two floats (K positions 2e, 2e+1) into packed bf16 hi and lo words
__device__ __forceinline__ void split2(float a, float b, uint32_t& hi, uint32_t& lo) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);  // a in the low half
    const __nv_bfloat162 l = __floats2bfloat162_rn(a - __low2float(h), b - __high2float(h));
    hi = *reinterpret_cast<const uint32_t*>(&h);
    lo = *reinterpret_cast<const uint32_t*>(&l);
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t mbar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_init_n(uint32_t mbar, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mbar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t mbar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar) : "memory");
}
// bounded wait with a caller-given limit
__device__ __forceinline__ bool mbar_wait_lim(uint32_t mbar, uint32_t parity, long long lim) {
    const long long t0 = clock64();
    while (true) {
        uint32_t ok;
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(mbar), "r"(parity)
            : "memory");
        if (ok) return true;
        if (clock64() - t0 > lim) return false;
    }
}

__device__ __forceinline__ void zero8(float2 (&v)[8]) {
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = make_float2(0.f, 0.f);
}

// Operand sources.  load_a(row, q, k0, v) fills the 8 values K = k0+8q.. of
// A row `row`; load_b(col, q, k0, v) those of right-hand side `col`.
struct Phase1 {
    // stacked rows of R (conj of the stored R^H rows) times x gathered over the source atoms
    const float2* fac;
    const long long* rowoff;
    const int* rowt;
    const int* S;
    const float2* x;
    int64_t ldx;
    int np, nK, row_begin, rows, c0, ncol;
    __device__ __forceinline__ void load_a(int row, int q, int k0, float2 (&v)[8]) const {
        const int j = k0 + 8 * q;
        if (row >= rows || j >= nK) {
            zero8(v);
            return;
        }
        const float2* src = fac + rowoff[row_begin + row] + j;
        if (j + 8 <= nK) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float4 w = __ldcs(reinterpret_cast<const float4*>(src) + e);
                v[2 * e] = make_float2(w.x, -w.y);
                v[2 * e + 1] = make_float2(w.z, -w.w);
            }
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float2 w = j + e < nK ? __ldcs(src + e) : make_float2(0.f, 0.f);
                v[e] = make_float2(w.x, -w.y);
            }
        }
    }
    __device__ __forceinline__ void load_b(int col, int q, int k0, float2 (&v)[8]) const {
        const int j = k0 + 8 * q;
        if (col >= ncol || j >= nK) {
            zero8(v);
            return;
        }
        const float2* xc = x + (int64_t)(c0 + col) * ldx;
        const int slot = j / np, off = j - slot * np;
        if (j + 8 <= nK && off + 8 <= np) {
            const float4* p = reinterpret_cast<const float4*>(xc + (int64_t)S[slot] * np + off);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float4 w = __ldg(p + e);
                v[2 * e] = make_float2(w.x, w.y);
                v[2 * e + 1] = make_float2(w.z, w.w);
            }
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int jj = j + e;
                if (jj < nK) {
                    const int sl = jj / np, of = jj - sl * np;
                    v[e] = __ldg(xc + (int64_t)S[sl] * np + of);
                } else {
                    v[e] = make_float2(0.f, 0.f);
                }
            }
        }
    }
};

}  // namespace vie
