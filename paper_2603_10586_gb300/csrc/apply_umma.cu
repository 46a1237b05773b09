// Multi-right-hand-side far apply on the 5th-generation tensor cores
// (tcgen05.mma, accumulators in tensor memory), split precision BF16x3.
//
// With s right-hand sides the far apply is two sets of dense contractions,
//   phase 1:  t_b = R_b X_J           (paper Sec. 5.2, the inner product R x)
//   phase 2:  F_a = sum_b Q_b[a] t_b  (the outer product Q t, per atom a)
// Each complex float32 operand value v is split into bfloat16 hi = bf16(v)
// and lo = bf16(v - hi) for its real and imaginary parts; a real product is
// hi.hi + hi.lo + lo.hi (the lo.lo term, ~2^-16 relative, is dropped), so a
// complex product is twelve bf16 MMAs accumulated in float32:
//   D_r += Ar Br - Ai Bi,   D_i += Ar Bi + Ai Br,
// the minus sign taken by the MMA's negate-A bit.
//
// Tile: 128 output rows (tensor-memory lanes) x up to 64 right-hand sides;
// D_r occupies tensor-memory columns [0, 64) and D_i columns [64, 128).
// The K dimension is staged 32 complex values at a time: the four warps load
// the operands from global memory, split them into bf16 planes and store the
// planes in shared memory in the canonical no-swizzle K-major layout (8x8
// core matrices of 128 contiguous bytes); one thread then issues the 24 MMAs
// of the stage and commits them to an mbarrier, and while the tensor core
// works on one stage the warps fill the other.
//
// Phase 1 stacks the R rows of all blocks that share one source atom list,
// so one gathered x_J feeds up to 128 rows; phase 2 walks one virtual K axis
// made of every (block, rank index) that touches the atom, so short ranks do
// not pad the K stages.
//
// Every wait on an mbarrier gives up after about a second of clock cycles,
// records the failure in an error word and leaves the kernel after freeing
// its tensor memory.
#include <cstdlib>
#include <mutex>

#include "common.h"
#include "cplx.cuh"
#include "umma.cuh"

namespace vie {

namespace {

constexpr int kM = 128;                 // output rows per tile
constexpr int kN = 64;                  // right-hand sides per pass
constexpr int kKS = 32;                 // complex K values per stage
constexpr int kThr = 256;               // eight warps (two per tensor-memory lane quarter)
constexpr int kTmemCols = 128;          // D_r: [0, 64), D_i: [64, 128)
constexpr int kChunksA = kM * kKS / 8;  // 16-byte chunks per A plane (512)
constexpr int kChunksB = kN * kKS / 8;  // 16-byte chunks per B plane (256)
constexpr uint32_t kLboA = kM * 16;     // bytes between K-adjacent core matrices of A
constexpr uint32_t kLboB = kN * 16;

// one stage: planes (re hi, re lo, im hi, im lo) of A (128 x 32) and B (64 x 32);
// chunk (row, q) of a plane holds K values 8q .. 8q+7 of that row and sits at
// index q * rows + row, i.e. core matrix (row / 8, q) at q * LBO + (row / 8) * 128
struct Stage {
    uint4 a[4][kChunksA];
    uint4 b[4][kChunksB];
};
constexpr size_t kStageBytes = sizeof(Stage);  // 48 KiB
constexpr size_t kSmemBytes = 2 * kStageBytes;  // two stages: 96 KiB, two CTAs per SM

// 8 complex values -> the 16-byte chunk of each plane
template <int CHUNKS>
__device__ __forceinline__ void put8(uint4 (*planes)[CHUNKS], int chunk, const float2 (&v)[8]) {
    uint32_t rh[4], rl[4], ih[4], il[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        split2(v[2 * e].x, v[2 * e + 1].x, rh[e], rl[e]);
        split2(v[2 * e].y, v[2 * e + 1].y, ih[e], il[e]);
    }
    planes[0][chunk] = make_uint4(rh[0], rh[1], rh[2], rh[3]);
    planes[1][chunk] = make_uint4(rl[0], rl[1], rl[2], rl[3]);
    planes[2][chunk] = make_uint4(ih[0], ih[1], ih[2], ih[3]);
    planes[3][chunk] = make_uint4(il[0], il[1], il[2], il[3]);
}

// the 24 MMAs of one stage (two K steps of 16)
__device__ __forceinline__ void issue_stage(const Stage& st, uint32_t tm, int nmma, bool first) {
    const uint32_t id = idesc(nmma, false), idn = idesc(nmma, true);
#pragma unroll
    for (int ks = 0; ks < 2; ++ks) {
        uint64_t A[4], B[4];
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            A[p] = sdesc(smem_u32(&st.a[p][0]) + ks * 2 * kLboA, kLboA);
            B[p] = sdesc(smem_u32(&st.b[p][0]) + ks * 2 * kLboB, kLboB);
        }
        const uint32_t acc0 = (first && ks == 0) ? 0u : 1u;
        // planes: 0 re hi, 1 re lo, 2 im hi, 3 im lo
        umma(tm, A[0], B[0], id, acc0);
        umma(tm, A[0], B[1], id, 1u);
        umma(tm, A[1], B[0], id, 1u);
        umma(tm, A[2], B[2], idn, 1u);
        umma(tm, A[2], B[3], idn, 1u);
        umma(tm, A[3], B[2], idn, 1u);
        umma(tm + kN, A[0], B[2], id, acc0);
        umma(tm + kN, A[0], B[3], id, 1u);
        umma(tm + kN, A[1], B[2], id, 1u);
        umma(tm + kN, A[2], B[0], id, 1u);
        umma(tm + kN, A[2], B[1], id, 1u);
        umma(tm + kN, A[3], B[0], id, 1u);
    }
}

struct Phase2 {
    // rows p0.. of one atom in every Q_b touching it, times the matching t_b entries
    const float2* fac;
    const long long* qoff;
    const int* tidx;
    const float2* t;
    int64_t ldt;
    int64_t kbase;
    int nK, p0, rows, c0, ncol;
    __device__ __forceinline__ void load_a(int row, int q, int k0, float2 (&v)[8]) const {
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int kk = k0 + 8 * q + e;
            v[e] = (row < rows && kk < nK) ? __ldcs(fac + qoff[kbase + kk] + p0 + row) : make_float2(0.f, 0.f);
        }
    }
    __device__ __forceinline__ void load_b(int col, int q, int k0, float2 (&v)[8]) const {
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const int kk = k0 + 8 * q + e;
            v[e] = (col < ncol && kk < nK) ? __ldg(t + tidx[kbase + kk] + (int64_t)(c0 + col) * ldt)
                                           : make_float2(0.f, 0.f);
        }
    }
};

// A segments: phase 1 keeps the 4 K chunks of a row on neighbouring threads
// (contiguous R rows), phase 2 keeps rows on neighbouring threads (contiguous
// Q columns)
template <bool kRowFast>
__device__ __forceinline__ void a_seg(int s, int& row, int& q) {  // s in [0, 512)
    if (kRowFast) {
        row = s & (kM - 1);
        q = s >> 7;
    } else {
        row = s >> 2;
        q = s & 3;
    }
}

struct Ctl {
    uint64_t mbar[2];  // MMAs of the stage in buffer b done
    uint64_t tma[2];   // packed variant: A of the stage in buffer b landed
    uint32_t tmem;
    int ok;
};

constexpr int kStageChunksA = 4 * kChunksA;      // 16-byte chunks of one packed A stage (2048)
constexpr uint32_t kStageBytesA = kStageChunksA * 16;  // 32 KiB

// bulk copy global -> shared memory, completion counted on the mbarrier.  The
// factor planes are read once per apply, so their lines are marked first to
// leave L2, in favour of the gathered x / t rows that many tiles read.
__device__ __forceinline__ uint64_t l2_evict_first_policy() {
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ void tma_bulk(uint32_t dst, const void* src, uint32_t bytes, uint32_t mbar) {
    const uint64_t pol = l2_evict_first_policy();
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::
            "r"(dst),
        "l"(src), "r"(bytes), "r"(mbar), "l"(pol)
        : "memory");
}

// One output tile (rows x ncol) over K = nK: stages g0, g0+1, ... of this CTA.
// Returns false when a wait gave up.  On return every thread may read the
// accumulators (when nK > 0).

template <class Src, bool kRowFast>
__device__ bool run_tile(const Src& src, Stage* stages, Ctl& ctl, uint32_t& g, int nK, int nmma) {
    const int tid = threadIdx.x;
    const int nst = (nK + kKS - 1) / kKS;
    for (int st = 0; st < nst; ++st, ++g) {
        const int k0 = st * kKS;
        Stage& S = stages[g & 1];
        // A: 512 segments of 8 values, B: 256 (two and one per thread)
        float2 va[2][8], vb[8];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            int row, q;
            a_seg<kRowFast>(tid + i * kThr, row, q);
            src.load_a(row, q, k0, va[i]);
        }
        src.load_b(tid >> 2, tid & 3, k0, vb);
        // the stage buffer is free once the MMAs issued two stages ago are done
        if (tid == 0) ctl.ok = (g < 2) ? 1 : (mbar_wait(smem_u32(&ctl.mbar[g & 1]), ((g >> 1) - 1) & 1) ? 1 : 0);
        __syncthreads();
        if (!ctl.ok) return false;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            int row, q;
            a_seg<kRowFast>(tid + i * kThr, row, q);
            put8<kChunksA>(S.a, q * kM + row, va[i]);
        }
        put8<kChunksB>(S.b, (tid & 3) * kN + (tid >> 2), vb);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (tid == 0) {
            fence_after();
            issue_stage(S, ctl.tmem, nmma, st == 0);
            umma_commit(smem_u32(&ctl.mbar[g & 1]));
        }
    }
    if (nst > 0) {
        const uint32_t gl = g - 1;
        if (tid == 0) ctl.ok = mbar_wait(smem_u32(&ctl.mbar[gl & 1]), (gl >> 1) & 1) ? 1 : 0;
        __syncthreads();
        if (!ctl.ok) return false;
        fence_after();
    }
    return true;
}

// The packed variant: the A operand of every stage is already split into bf16
// planes in the stage layout (packA, 32 KiB per stage), so one thread moves
// it with a bulk copy, one stage ahead, while the warps split only B.
// `alive` (thread 0's) turns false when a wait gave up.
__device__ __forceinline__ void issue_a(Ctl& ctl, Stage* stages, uint32_t g, const uint4* src) {
    const uint32_t mb = smem_u32(&ctl.tma[g & 1]);
    mbar_expect_tx(mb, kStageBytesA);
    tma_bulk(smem_u32(&stages[g & 1].a[0][0]), src, kStageBytesA, mb);
}

template <class Src>
__device__ bool run_tile_tma(const Src& src, const uint4* packA, Stage* stages, Ctl& ctl, uint32_t& g, int nK,
                             int nmma, bool& alive) {
    const int tid = threadIdx.x;
    const int nst = (nK + kKS - 1) / kKS;
    for (int st = 0; st < nst; ++st, ++g) {
        Stage& S = stages[g & 1];
        float2 vb[8];
        src.load_b(tid >> 2, tid & 3, st * kKS, vb);
        if (tid == 0) {
            // a buffer is free once the MMAs issued two stages before it are done
            if (st == 0 && alive) {
                if (g >= 2) alive = mbar_wait(smem_u32(&ctl.mbar[g & 1]), ((g >> 1) - 1) & 1);
                if (alive) issue_a(ctl, stages, g, packA);
            }
            if (st + 1 < nst && alive) {
                const uint32_t g1 = g + 1;
                if (g1 >= 2) alive = mbar_wait(smem_u32(&ctl.mbar[g1 & 1]), ((g1 >> 1) - 1) & 1);
                if (alive) issue_a(ctl, stages, g1, packA + (int64_t)(st + 1) * kStageChunksA);
            }
            ctl.ok = alive ? 1 : 0;
        }
        __syncthreads();
        if (!ctl.ok) return false;
        put8<kChunksB>(S.b, (tid & 3) * kN + (tid >> 2), vb);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (tid == 0 && alive) {
            alive = mbar_wait(smem_u32(&ctl.tma[g & 1]), (g >> 1) & 1);
            if (alive) {
                fence_after();
                issue_stage(S, ctl.tmem, nmma, st == 0);
                umma_commit(smem_u32(&ctl.mbar[g & 1]));
            }
        }
    }
    if (nst > 0) {
        const uint32_t gl = g - 1;
        if (tid == 0) {
            if (alive) alive = mbar_wait(smem_u32(&ctl.mbar[gl & 1]), (gl >> 1) & 1);
            ctl.ok = alive ? 1 : 0;
        }
        __syncthreads();
        if (!ctl.ok) return false;
        fence_after();
    }
    return true;
}

// out[rowidx(r) + c * ld] = (D_r, D_i)[r, c] for r < rows, c < ncol (zeros when nK == 0).
// A warp reads the tensor-memory lanes of its quarter (warp % 4); warps 0-3
// take columns 0-31, warps 4-7 columns 32-63.
template <class RowIdx>
__device__ void epilogue(const Ctl& ctl, bool have, int rows, int ncol, RowIdx rowidx, float2* out, int64_t ld) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int quarter = warp & 3, half = warp >> 2;
    const int r = quarter * 32 + lane;
    const uint32_t base = ctl.tmem + ((uint32_t)(quarter * 32) << 16);
    const bool mine = r < rows;
    const int64_t ri = mine ? rowidx(r) : 0;
    for (int cb = half * 32; cb < min(ncol, half * 32 + 32); cb += 16) {
        float vr[16], vi[16];
        if (have) {
            tmem_ld16(base + cb, vr);
            tmem_ld16(base + kN + cb, vi);
            tmem_wait_ld();
        } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) vr[i] = vi[i] = 0.f;
        }
        if (mine) {
#pragma unroll
            for (int i = 0; i < 16; ++i)
                if (cb + i < ncol) out[ri + (int64_t)(cb + i) * ld] = make_float2(vr[i], vi[i]);
        }
    }
    fence_before();
    __syncthreads();  // accumulators read before the next tile overwrites them
}

__device__ void setup(Ctl& ctl) {
    if (threadIdx.x == 0) {
        mbar_init(smem_u32(&ctl.mbar[0]));
        mbar_init(smem_u32(&ctl.mbar[1]));
        mbar_init(smem_u32(&ctl.tma[0]));
        mbar_init(smem_u32(&ctl.tma[1]));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if ((threadIdx.x >> 5) == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl.tmem)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
}

// leave: if a wait gave up, give the tensor core one more bounded chance to
// finish what was issued, then free the tensor memory
__device__ void teardown(Ctl& ctl, bool failed, uint32_t g, int* err) {
    if (failed) {
        if (threadIdx.x == 0) {
            atomicExch(err, 1);
            if (g > 0) mbar_wait(smem_u32(&ctl.mbar[(g - 1) & 1]), ((g - 1) >> 1) & 1);
        }
    }
    fence_before();
    __syncthreads();
    fence_after();
    if ((threadIdx.x >> 5) == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(ctl.tmem), "r"(kTmemCols)
                     : "memory");
}

__global__ void __launch_bounds__(kThr) u1_kernel(const FarBlockDev* __restrict__ blocks,
                                                  const int* __restrict__ batoms, const int4* __restrict__ items,
                                                  const int* __restrict__ cta_ptr,
                                                  const long long* __restrict__ rowoff, const int* __restrict__ rowt,
                                                  const float2* __restrict__ fac, const float2* __restrict__ x,
                                                  int64_t ldx, int np, float2* __restrict__ t, int64_t ldt, int nrhs,
                                                  const int2* __restrict__ colr, int* err) {
    extern __shared__ __align__(1024) unsigned char smem[];
    Stage* stages = reinterpret_cast<Stage*>(smem);
    __shared__ Ctl ctl;
    setup(ctl);
    uint32_t g = 0;
    bool failed = false;
    for (int it = cta_ptr[blockIdx.x]; it < cta_ptr[blockIdx.x + 1] && !failed; ++it) {
        const int4 item = items[it];
        const FarBlockDev B = blocks[item.x];
        const int2 cr = colr ? colr[item.w] : make_int2(0, nrhs);  // right-hand sides of this problem
        for (int c0 = cr.x; c0 < cr.y && !failed; c0 += kN) {
            Phase1 src{fac, rowoff, rowt, batoms + B.s_off, x, ldx, np, B.n, item.y, item.z, c0, min(kN, cr.y - c0)};
            const int nmma = max(16, (src.ncol + 15) / 16 * 16);
            if (!run_tile<Phase1, false>(src, stages, ctl, g, B.n, nmma)) {
                failed = true;
                break;
            }
            const int* rt = rowt + item.y;
            epilogue(ctl, B.n > 0, item.z, src.ncol, [rt](int r) { return (int64_t)rt[r]; }, t + (int64_t)c0 * ldt,
                     ldt);
        }
    }
    teardown(ctl, failed, g, err);
}

__global__ void __launch_bounds__(kThr) u2_kernel(const int4* __restrict__ items, const int* __restrict__ cta_ptr,
                                                  const long long* __restrict__ qoff, const int* __restrict__ tidx,
                                                  const long long* __restrict__ kptr, const float2* __restrict__ fac,
                                                  const float2* __restrict__ t, int64_t ldt, int np,
                                                  float2* __restrict__ F, int64_t ldf, int nrhs,
                                                  const int2* __restrict__ colr, int* err) {
    extern __shared__ __align__(1024) unsigned char smem[];
    Stage* stages = reinterpret_cast<Stage*>(smem);
    __shared__ Ctl ctl;
    setup(ctl);
    uint32_t g = 0;
    bool failed = false;
    for (int it = cta_ptr[blockIdx.x]; it < cta_ptr[blockIdx.x + 1] && !failed; ++it) {
        const int4 item = items[it];
        const int a = item.x, p0 = item.y, rows = item.z - item.y;
        const long long kb = kptr[a];
        const int nK = (int)(kptr[a + 1] - kb);
        const int2 cr = colr ? colr[item.w] : make_int2(0, nrhs);
        for (int c0 = cr.x; c0 < cr.y && !failed; c0 += kN) {
            Phase2 src{fac, qoff, tidx, t, ldt, kb, nK, p0, rows, c0, min(kN, cr.y - c0)};
            const int nmma = max(16, (src.ncol + 15) / 16 * 16);
            if (!run_tile<Phase2, true>(src, stages, ctl, g, nK, nmma)) {
                failed = true;
                break;
            }
            const int64_t rb = (int64_t)a * np + p0;
            epilogue(ctl, nK > 0, rows, src.ncol, [rb](int r) { return rb + r; }, F + (int64_t)c0 * ldf, ldf);
        }
    }
    teardown(ctl, failed, g, err);
}

// ---- packed variant ---------------------------------------------------------
// pack: one CTA per work item writes the item's A operand, stage after stage,
// in the shared-memory stage layout (zero padding past the last row / K value)
__global__ void __launch_bounds__(kThr) pack1_kernel(const FarBlockDev* __restrict__ blocks,
                                                     const int4* __restrict__ items, const long long* __restrict__ pk,
                                                     const long long* __restrict__ rowoff,
                                                     const float2* __restrict__ fac, int np, uint4* __restrict__ out) {
    const int4 item = items[blockIdx.x];
    const FarBlockDev B = blocks[item.x];
    const Phase1 src{fac, rowoff, nullptr, nullptr, nullptr, 0, np, B.n, item.y, item.z, 0, 0};
    const int nst = (B.n + kKS - 1) / kKS;
    uint4* base = out + pk[blockIdx.x] * kStageChunksA;
    for (int st = 0; st < nst; ++st) {
        uint4(*planes)[kChunksA] = reinterpret_cast<uint4(*)[kChunksA]>(base + (int64_t)st * kStageChunksA);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            int row, q;
            a_seg<false>(threadIdx.x + i * kThr, row, q);
            float2 v[8];
            src.load_a(row, q, st * kKS, v);
            put8<kChunksA>(planes, q * kM + row, v);
        }
    }
}

__global__ void __launch_bounds__(kThr) pack2_kernel(const int4* __restrict__ items, const long long* __restrict__ pk,
                                                     const long long* __restrict__ qoff,
                                                     const long long* __restrict__ kptr,
                                                     const float2* __restrict__ fac, uint4* __restrict__ out) {
    const int4 item = items[blockIdx.x];
    const int a = item.x;
    const long long kb = kptr[a];
    const int nK = (int)(kptr[a + 1] - kb);
    const Phase2 src{fac, qoff, nullptr, nullptr, 0, kb, nK, item.y, item.z - item.y, 0, 0};
    const int nst = (nK + kKS - 1) / kKS;
    uint4* base = out + pk[blockIdx.x] * kStageChunksA;
    for (int st = 0; st < nst; ++st) {
        uint4(*planes)[kChunksA] = reinterpret_cast<uint4(*)[kChunksA]>(base + (int64_t)st * kStageChunksA);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            int row, q;
            a_seg<true>(threadIdx.x + i * kThr, row, q);
            float2 v[8];
            src.load_a(row, q, st * kKS, v);
            put8<kChunksA>(planes, q * kM + row, v);
        }
    }
}

__global__ void __launch_bounds__(kThr) u1p_kernel(const FarBlockDev* __restrict__ blocks,
                                                   const int* __restrict__ batoms, const int4* __restrict__ items,
                                                   const int* __restrict__ cta_ptr, const long long* __restrict__ pk,
                                                   const uint4* __restrict__ pack, const int* __restrict__ rowt,
                                                   const float2* __restrict__ x, int64_t ldx, int np,
                                                   float2* __restrict__ t, int64_t ldt, int nrhs,
                                                   const int2* __restrict__ colr, int* err) {
    extern __shared__ __align__(1024) unsigned char smem[];
    Stage* stages = reinterpret_cast<Stage*>(smem);
    __shared__ Ctl ctl;
    setup(ctl);
    uint32_t g = 0;
    bool failed = false, alive = true;
    for (int it = cta_ptr[blockIdx.x]; it < cta_ptr[blockIdx.x + 1] && !failed; ++it) {
        const int4 item = items[it];
        const FarBlockDev B = blocks[item.x];
        const int2 cr = colr ? colr[item.w] : make_int2(0, nrhs);
        for (int c0 = cr.x; c0 < cr.y && !failed; c0 += kN) {
            Phase1 src{nullptr, nullptr, rowt, batoms + B.s_off, x, ldx, np, B.n, item.y, item.z, c0,
                       min(kN, cr.y - c0)};
            const int nmma = max(16, (src.ncol + 15) / 16 * 16);
            if (!run_tile_tma(src, pack + pk[it] * kStageChunksA, stages, ctl, g, B.n, nmma, alive)) {
                failed = true;
                break;
            }
            const int* rt = rowt + item.y;
            epilogue(ctl, B.n > 0, item.z, src.ncol, [rt](int r) { return (int64_t)rt[r]; }, t + (int64_t)c0 * ldt,
                     ldt);
        }
    }
    teardown(ctl, failed, g, err);
}

__global__ void __launch_bounds__(kThr) u2p_kernel(const int4* __restrict__ items, const int* __restrict__ cta_ptr,
                                                   const long long* __restrict__ pk, const uint4* __restrict__ pack,
                                                   const int* __restrict__ tidx, const long long* __restrict__ kptr,
                                                   const float2* __restrict__ t, int64_t ldt, int np,
                                                   float2* __restrict__ F, int64_t ldf, int nrhs,
                                                   const int2* __restrict__ colr, int* err) {
    extern __shared__ __align__(1024) unsigned char smem[];
    Stage* stages = reinterpret_cast<Stage*>(smem);
    __shared__ Ctl ctl;
    setup(ctl);
    uint32_t g = 0;
    bool failed = false, alive = true;
    for (int it = cta_ptr[blockIdx.x]; it < cta_ptr[blockIdx.x + 1] && !failed; ++it) {
        const int4 item = items[it];
        const int a = item.x, p0 = item.y, rows = item.z - item.y;
        const long long kb = kptr[a];
        const int nK = (int)(kptr[a + 1] - kb);
        const int2 cr = colr ? colr[item.w] : make_int2(0, nrhs);
        for (int c0 = cr.x; c0 < cr.y && !failed; c0 += kN) {
            Phase2 src{nullptr, nullptr, tidx, t, ldt, kb, nK, p0, rows, c0, min(kN, cr.y - c0)};
            const int nmma = max(16, (src.ncol + 15) / 16 * 16);
            if (!run_tile_tma(src, pack + pk[it] * kStageChunksA, stages, ctl, g, nK, nmma, alive)) {
                failed = true;
                break;
            }
            const int64_t rb = (int64_t)a * np + p0;
            epilogue(ctl, nK > 0, rows, src.ncol, [rb](int r) { return rb + r; }, F + (int64_t)c0 * ldf, ldf);
        }
    }
    teardown(ctl, failed, g, err);
}

std::once_flag g_umma_attr_once;

}  // namespace

void umma_prepare(Op& op, cudaStream_t s) {
    if (op.fprec != VIE_C64) fail(VIE_ERR_INVALID_ARG, "the tcgen05 apply needs VIE_C64 factors");
    build_umma_lists(op);
    std::call_once(g_umma_attr_once, [] {
        cudaFuncSetAttribute(u1_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
        cudaFuncSetAttribute(u2_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
        cudaFuncSetAttribute(u1p_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
        cudaFuncSetAttribute(u2p_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
    });
    if (!op.d_err.p) {
        op.d_err.alloc(sizeof(int));
        VIE_CUDA(cudaMemsetAsync(op.d_err.p, 0, sizeof(int), s));
    }
}

void apply_far_umma(Op& op, const float2* x, int64_t ldx, float2* F, int64_t ldf, int nrhs, cudaStream_t s) {
    umma_prepare(op, s);
    if (((uintptr_t)x & 15) || (ldx & 1)) fail(VIE_ERR_INVALID_ARG, "tensor-core apply: x must be 16-byte aligned");
    const size_t need = (size_t)std::max<int64_t>(op.t_total, 1) * nrhs * sizeof(float2);
    if (op.d_t.bytes < need) op.d_t.alloc(need);
    const float2* fac = op.fac<float2>();
    if (op.n_u1_items > 0) {
        u1_kernel<<<op.n_cta_u, kThr, kSmemBytes, s>>>(
            op.d_blocks.as<FarBlockDev>(), op.d_block_atoms.as<int>(), op.d_u1_items.as<int4>(), op.d_u1_cta.as<int>(),
            op.d_u1_rowoff.as<long long>(), op.d_u1_rowt.as<int>(), fac, x, ldx, op.np, op.d_t.as<float2>(),
            op.t_total, nrhs, op.colr, op.d_err.as<int>());
        VIE_CHECK_LAUNCH();
    }
    u2_kernel<<<op.n_cta_u, kThr, kSmemBytes, s>>>(
        op.d_u2_items.as<int4>(), op.d_u2_cta.as<int>(), op.d_u2_qoff.as<long long>(), op.d_u2_tidx.as<int>(),
        op.d_u2_kptr.as<long long>(), fac, op.d_t.as<float2>(), op.t_total, op.np, F, ldf, nrhs, op.colr,
        op.d_err.as<int>());
    VIE_CHECK_LAUNCH();
}

size_t umma_pack_bytes(const Op& op) { return (size_t)(op.u1_stages + op.u2_stages) * kStageBytesA; }

bool umma_pack(Op& op, cudaStream_t s) {
    umma_prepare(op, s);
    if (op.umma_packed) return true;
    if (op.umma_pack_failed) return false;
    const size_t b1 = (size_t)op.u1_stages * kStageBytesA, b2 = (size_t)op.u2_stages * kStageBytesA;
    size_t free_b = 0, total_b = 0;
    VIE_CUDA(cudaMemGetInfo(&free_b, &total_b));
    if (b1 + b2 + ((size_t)1 << 30) > free_b) {  // keep 1 GiB for the solver
        op.umma_pack_failed = true;
        return false;
    }
    op.d_u1_pack.alloc(std::max<size_t>(b1, 16));
    op.d_u2_pack.alloc(std::max<size_t>(b2, 16));
    if (op.n_u1_items > 0) {
        pack1_kernel<<<op.n_u1_items, kThr, 0, s>>>(op.d_blocks.as<FarBlockDev>(), op.d_u1_items.as<int4>(),
                                                    op.d_u1_pk.as<long long>(), op.d_u1_rowoff.as<long long>(),
                                                    op.fac<float2>(), op.np, op.d_u1_pack.as<uint4>());
        VIE_CHECK_LAUNCH();
    }
    if (op.n_u2_items > 0) {
        pack2_kernel<<<op.n_u2_items, kThr, 0, s>>>(op.d_u2_items.as<int4>(), op.d_u2_pk.as<long long>(),
                                                    op.d_u2_qoff.as<long long>(), op.d_u2_kptr.as<long long>(),
                                                    op.fac<float2>(), op.d_u2_pack.as<uint4>());
        VIE_CHECK_LAUNCH();
    }
    op.umma_packed = true;
    return true;
}

void apply_far_umma_packed(Op& op, const float2* x, int64_t ldx, float2* F, int64_t ldf, int nrhs, cudaStream_t s) {
    if (!umma_pack(op, s)) {  // not enough memory for the packed planes: the kernel that splits A itself
        apply_far_umma(op, x, ldx, F, ldf, nrhs, s);
        return;
    }
    if (((uintptr_t)x & 15) || (ldx & 1)) fail(VIE_ERR_INVALID_ARG, "tensor-core apply: x must be 16-byte aligned");
    const size_t need = (size_t)std::max<int64_t>(op.t_total, 1) * nrhs * sizeof(float2);
    if (op.d_t.bytes < need) op.d_t.alloc(need);
    if (op.n_u1_items > 0) {
        u1p_kernel<<<op.n_cta_u, kThr, kSmemBytes, s>>>(
            op.d_blocks.as<FarBlockDev>(), op.d_block_atoms.as<int>(), op.d_u1_items.as<int4>(), op.d_u1_cta.as<int>(),
            op.d_u1_pk.as<long long>(), op.d_u1_pack.as<uint4>(), op.d_u1_rowt.as<int>(), x, ldx, op.np,
            op.d_t.as<float2>(), op.t_total, nrhs, op.colr, op.d_err.as<int>());
        VIE_CHECK_LAUNCH();
    }
    u2p_kernel<<<op.n_cta_u, kThr, kSmemBytes, s>>>(
        op.d_u2_items.as<int4>(), op.d_u2_cta.as<int>(), op.d_u2_pk.as<long long>(), op.d_u2_pack.as<uint4>(),
        op.d_u2_tidx.as<int>(), op.d_u2_kptr.as<long long>(), op.d_t.as<float2>(), op.t_total, op.np, F, ldf, nrhs,
        op.colr, op.d_err.as<int>());
    VIE_CHECK_LAUNCH();
}

}  // namespace vie
