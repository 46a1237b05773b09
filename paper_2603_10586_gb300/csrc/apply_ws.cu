// Multi-right-hand-side far apply on the 5th-generation tensor cores (tcgen05.mma,
// accumulators in tensor memory), split precision BF16x3, warp-specialised and
// persistent (variants 9 and 10; apply_umma.cu has the arithmetic and the plain
// kernels).
//
// The two products are those of apply_umma.cu,
//   phase 1:  t_b = R_b X_J           for the stacked rows of every block with source box J
//   phase 2:  F_a = sum_b Q_b[a] t_b  along one K axis over every block of atom a,
// with every factor split once into bf16 planes (re hi, re lo, im hi, im lo).  The
// planes are held once per factor storage: the tiles of translated copies read
// the same planes, so the operand that used to stream from HBM for every block
// (19.7 GB per product of the 32 x 32 array of 4^3 cubes, 72-97% of the HBM rate)
// is 0.93 GB that mostly stays in L2.  For that the planes are cut where blocks
// end, at 8 rows of R and 8 columns of Q:
//   R: per 16 K values and 8 rows one kilobyte, [plane][K / 8][row] of 16-byte
//      chunks; a tile of 128 stacked rows is a few runs of consecutive groups, one
//      bulk copy each;
//   Q: per 8 K values and 128 rows of one target slot 8 KB, [plane][row], the
//      chunks of a block and slot in a row; a stage takes the chunks of its K
//      values, whatever blocks they belong to.
// Ranks are padded to 8 (with zeros), and so is t, which lies as [eight K values]
// [column][K value]: the 64 columns of a chunk are 4 KB in a row.  (Column after
// column, 18 MB apart on the 32 x 32 array, every chunk touched 64 pages.)
//
// One persistent CTA per SM; the roles run concurrently and meet on mbarriers
// instead of CTA-wide barriers:
//   warp 4     starts the bulk copies of the A planes of every K stage (32 KiB)
//              into the next free slot of a ring of 4 to 6 stages (as many as fit
//              beside the B planes of the widest tile), a lane per copy;
//   warps 5-12 four groups of two warps (never more than the ring has
//              stages) load, split and store the B operand (x gathered over
//              the source atoms, or t) of a stage; group q takes the stages
//              g = q mod 4 and gathers a stage's values into registers before
//              it waits for the stage's slot, so the loads of four stages are in
//              flight while the MMAs run;
//   warp 13    one elected lane issues the 8 MMAs of a stage once its A copies have
//              landed and its B planes are stored, and commits them to the
//              slot's "empty" barrier (the producers refill it) and, at the end
//              of a tile, to the tile's accumulator barrier;
//   warps 0-3  epilogue: read the finished tile from tensor memory (warp w
//              owns lanes 32w..32w+31) and store it.  Tensor memory holds two
//              accumulator buffers, so the MMAs of the next tile run while the
//              previous one drains.
// With B stored as two stacks of planes, S1 = [Br_hi; Bi_hi; Br_lo; Bi_lo] and
// S2 = [-Bi_hi; Br_hi; -Bi_lo; Br_lo] (N = ncol rows each; the negation is exact
// in bf16), a K step is four MMAs into one accumulator of 4 ncol columns
// [Re_a | Im_a | Re_b | Im_b]:
//   Ar_hi x S1 (N = 4 ncol), Ai_hi x S2 (4 ncol), Ar_lo x S1[0:2 ncol],
//   Ai_lo x S2[0:2 ncol],
// and the epilogue adds Re = Re_a + Re_b, Im = Im_a + Im_b.  The products are
// those of the twelve-MMA form (hi.hi + hi.lo + lo.hi of every real product);
// each A plane is read by one MMA.  The float32 sums are grouped differently, so
// the results agree with apply_umma.cu to rounding.
// What bounds it (16 columns on the graded 24 x 24 array, 64 on the 32 x 32 array,
// both of 4^3 cubes): the A planes pass from L2 to the SMs at 9.5 TB/s per phase,
// 32 KB per stage whatever the columns; with the planes hot in L2 and no B
// gathers the phases still take 85% of their time, with the MMAs left out 80-97%.
// Measured, phase 1 + phase 2: 724 + 709 -> 534 + 508 us (graded), 2048 + 2135 ->
// 1423 + 1213 us and 0.06 ms for x8 (32 x 32).
// Every wait gives up after `lim` clock cycles: the waiting role raises the
// CTA's abort flag, every role leaves its loop at its next check, and before
// the tensor memory is freed and the CTA exits, the bulk copies that were
// started and the MMAs that were issued are waited for (with the normal ~1 s
// limit).  The error word then tells the host.
#include <mutex>

#include "common.h"
#include "cplx.cuh"
#include "umma.cuh"

namespace vie {

namespace {

constexpr int kM = 128;   // output rows per tile
constexpr int kN = 64;    // right-hand sides per pass
constexpr int kWsMaxStages = 6;
constexpr int kWsThr = 448;  // 14 warps
constexpr int kWsWarpTma = 4, kWsWarpB0 = 5, kWsWarpMma = 13;
constexpr int kWsGroups = (kWsWarpMma - kWsWarpB0) / 2;  // B-producer groups of two warps
constexpr int kWsTmemCols = 512;                          // accumulators [Re_a | Im_a | Re_b | Im_b] of 4 nmax columns
constexpr int kWsSmemBytes = 224 * 1024;                  // the ring

// A planes in a stage: 16 KB units of 16 K values x 128 rows.  Phase 1: 16 groups
// of 8 rows, [plane][K / 8][row]; phase 2: two 8 KB chunks of 8 K values,
// [plane][row].  Byte offsets of a plane, of K-adjacent core matrices, of 8-row
// groups.
constexpr uint32_t kUnit = 16384;
template <int PHASE>
struct APlanes {
    static constexpr uint32_t plane = PHASE == 1 ? 256 : 2048;
    static constexpr uint32_t lbo = PHASE == 1 ? 128 : 8192;
    static constexpr uint32_t sbo = PHASE == 1 ? 1024 : 128;
};

// Two tile shapes share the code.  MT = 1: one 128-row M tile per B tile and
// 32 K values per stage (two units of 16).  MT = 2: two M tiles (256 rows: the
// two row tiles of one target atom, or two consecutive row tiles of one
// source group) share one B tile, 16 K values per stage (a unit per tile), so
// the B operand is gathered and split once for twice the factor rows.  Either way
// a stage carries 32 KiB of A planes.
template <int MT>
struct WsGeom {
    static constexpr int KS = 32 / MT;      // K values per stage
    static constexpr int KQ = KS / 8;       // 16-byte K chunks per row and stage
    static constexpr int KSTEPS = KS / 16;  // MMA K steps per stage
    static constexpr uint32_t kABytes = 2 * kUnit;
    // stage bytes: the A planes, then two B stacks of 4 KQ nmax chunks
    __host__ __device__ static constexpr uint32_t stride(int nmax) { return kABytes + 2u * 4u * KQ * nmax * 16u; }
    __host__ __device__ static constexpr int stages(int nmax) {
        return (int)(kWsSmemBytes / stride(nmax)) < kWsMaxStages ? (int)(kWsSmemBytes / stride(nmax)) : kWsMaxStages;
    }
    // accumulator buffers: each holds MT accumulators of 4 nmax columns
    __host__ __device__ static constexpr int nbuf(int nmax) { return kWsTmemCols / (MT * 4 * nmax) >= 2 ? 2 : 1; }
};
static_assert(WsGeom<1>::stages(32) == 4 && WsGeom<1>::stages(16) == 5, "ring sizes");
static_assert(WsGeom<2>::stages(64) == 4 && WsGeom<2>::stages(16) == 6, "ring sizes");
static_assert(WsGeom<2>::stride(16) % 1024 == 0 && WsGeom<1>::stride(16) % 1024 == 0, "stage alignment");

// The ring: ns stages of `stride` bytes.  A stage holds the A planes, then the
// two B stacks; chunk (slot, row, q) of a stack sits at q (4 nmma) + slot nmma
// + row.  nmax, the widest tile's column count rounded up to 16, sets the
// stride, and the stage count is what fits: for MT = 1 (up to 32 columns), 5
// stages up to 16 right-hand sides, else 4; for MT = 2, 6 up to 16, 5 up to 48, 4 up to 64.
struct WsRing {
    unsigned char* base;
    uint32_t stride, bstack;  // bytes per stage; chunks per B stack
    uint32_t ns;              // stages
    __device__ __forceinline__ uint32_t a(uint32_t slot) const { return smem_u32(base + slot * stride); }
    __device__ __forceinline__ uint4* b(uint32_t slot, int k) const {
        return reinterpret_cast<uint4*>(base + slot * stride + 2 * kUnit) + k * bstack;
    }
};
template <int MT>
__device__ __forceinline__ WsRing ws_ring(unsigned char* smem, int nmax) {
    return WsRing{smem, WsGeom<MT>::stride(nmax), 4u * WsGeom<MT>::KQ * nmax, (uint32_t)WsGeom<MT>::stages(nmax)};
}

__device__ __forceinline__ uint4 neg_bf16x8(uint4 v) {
    return make_uint4(v.x ^ 0x80008000u, v.y ^ 0x80008000u, v.z ^ 0x80008000u, v.w ^ 0x80008000u);
}

// the four planes' 16-byte chunks of 8 complex values
struct Chunks {
    uint4 rh, rl, ih, il;
};
__device__ __forceinline__ Chunks split8(const float2 (&v)[8]) {
    uint32_t rh[4], rl[4], ih[4], il[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        split2(v[2 * e].x, v[2 * e + 1].x, rh[e], rl[e]);
        split2(v[2 * e].y, v[2 * e + 1].y, ih[e], il[e]);
    }
    return {make_uint4(rh[0], rh[1], rh[2], rh[3]), make_uint4(rl[0], rl[1], rl[2], rl[3]),
            make_uint4(ih[0], ih[1], ih[2], ih[3]), make_uint4(il[0], il[1], il[2], il[3])};
}

// 8 complex values of B (column `row`, K chunk q) into both stacks
__device__ __forceinline__ void put8_ws(uint4* b0, uint4* b1, int nmma, int row, int q, const Chunks& c) {
    const int base = q * 4 * nmma + row;
    b0[base] = c.rh;
    b0[base + nmma] = c.ih;
    b0[base + 2 * nmma] = c.rl;
    b0[base + 3 * nmma] = c.il;
    b1[base] = neg_bf16x8(c.ih);
    b1[base + nmma] = c.rh;
    b1[base + 2 * nmma] = neg_bf16x8(c.il);
    b1[base + 3 * nmma] = c.rl;
}

// One MMA with its descriptors given as words: the low word is (address >> 4) |
// (LBO >> 4) << 16, and addresses stay below 2^18, so a descriptor moves by
// adding (bytes >> 4) to its low word.  The issuing thread is a serial resource:
// with descriptors, ring positions and timers recomputed per stage it took ~1,500
// cycles per stage, twice the tensor core's time.
__device__ __forceinline__ void umma_w(uint32_t dt, uint32_t alo, uint32_t ahi, uint32_t blo, uint32_t bhi, uint32_t id,
                                       uint32_t acc) {
    asm volatile(
        "{\n.reg .pred p;\n.reg .b64 da, db;\nsetp.ne.b32 p, %6, 0;\nmov.b64 da, {%1, %2};\nmov.b64 db, {%3, %4};\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;\n}\n" ::"r"(dt),
        "r"(alo), "r"(ahi), "r"(blo), "r"(bhi), "r"(id), "r"(acc));
}
constexpr uint32_t desc_hi(uint32_t sbo) { return (sbo >> 4) | (1u << 14); }  // SBO, descriptor version

// the four wide MMAs of one K step (16): A unit and B stacks at the given low
// words (without LBO), accumulator at tm
template <int PHASE>
__device__ __forceinline__ void mma_kstep_ws(uint32_t a, uint32_t b0, uint32_t b1, uint32_t tm, uint32_t id4,
                                             uint32_t id2, uint32_t acc0) {
    using P = APlanes<PHASE>;
    constexpr uint32_t ah = desc_hi(P::sbo), bh = desc_hi(128), l = (P::lbo >> 4) << 16, p = P::plane >> 4;
    // planes: 0 re hi, 1 re lo, 2 im hi, 3 im lo
    umma_w(tm, a + l, ah, b0, bh, id4, acc0);
    umma_w(tm, a + l + 2 * p, ah, b1, bh, id4, 1u);
    umma_w(tm, a + l + p, ah, b0, bh, id2, 1u);
    umma_w(tm, a + l + 3 * p, ah, b1, bh, id2, 1u);
}

// position in the ring: slot, and the parity of the pass over it
struct RingPos {
    uint32_t slot = 0, par = 0;
    __device__ __forceinline__ void step(uint32_t by, uint32_t ns) {  // by <= ns
        slot += by;
        if (slot >= ns) {
            slot -= ns;
            par ^= 1;
        }
    }
};

// bulk copy global -> shared memory, completion counted on the mbarrier
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void* src, uint32_t bytes, uint32_t mbar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(mbar)
                 : "memory");
}

struct WsCtl {
    uint64_t full_a[kWsMaxStages];  // A copies of the slot landed (1 arrival + bytes)
    uint64_t full_b[kWsMaxStages];  // B planes of the slot stored (the stage's 2 producer warps)
    uint64_t empty[kWsMaxStages];   // MMAs that read the slot are done (1 commit)
    uint64_t acc_full[2];        // accumulator buffer holds a finished tile (1 commit)
    uint64_t acc_empty[2];       // epilogue has read the buffer (4 epilogue warps)
    uint32_t tmem;
    volatile int abort;
    uint32_t g_tma, g_mma;       // stages whose A copies were started / whose MMAs were issued
};

__device__ __forceinline__ bool mbar_try(uint32_t mbar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(mbar), "r"(parity)
        : "memory");
    return ok != 0;
}
// wait for the phase with the given parity, at most `lim` cycles and not beyond
// an abort; the timer starts only when the first try fails (a limit of 0 gives up there)
__device__ __forceinline__ bool ws_wait(WsCtl& ctl, uint64_t& bar, uint32_t parity, long long lim) {
    const uint32_t mb = smem_u32(&bar);
    if (mbar_try(mb, parity)) return true;
    const long long t0 = clock64();
    while (!ctl.abort) {
        if (clock64() - t0 >= lim) {
            ctl.abort = 1;
            return false;
        }
        if (mbar_try(mb, parity)) return true;
    }
    return false;
}

// the same by a whole warp, with one answer for all lanes
__device__ __forceinline__ bool ws_wait_warp(WsCtl& ctl, uint64_t& bar, uint32_t parity, long long lim) {
    if (__all_sync(0xffffffffu, mbar_try(smem_u32(&bar), parity))) return true;
    const bool ok = ws_wait(ctl, bar, parity, lim);
    return __all_sync(0xffffffffu, ok);
}
__device__ __forceinline__ bool elect_one() {
    uint32_t e;
    asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}\n" : "=r"(e));
    return e != 0;
}

// ---- the tiles of a CTA, in the same order for every role --------------------
// (item, 64-column pass).  nst = K stages (0: nothing to multiply, the output is
// zero); nt = M tiles.
// One lane's copy of a stage: src + (stage) step, `bytes` to the stage's A
// planes + dst; bytes = 0: none.
struct WsCopy {
    const unsigned char* src;
    int64_t step;
    uint32_t dst, bytes;
};

// eight consecutive values
__device__ __forceinline__ void load8(const float2* src, float2 (&v)[8]) {
    const float4* p = reinterpret_cast<const float4*>(src);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float4 w = __ldg(p + e);
        v[2 * e] = make_float2(w.x, w.y);
        v[2 * e + 1] = make_float2(w.z, w.w);
    }
}

struct WsTile1 {
    struct Src {
        const int* S;      // source atoms
        const float2* x8;  // [chunk of an atom][column][8]
        int64_t ldx;       // values per chunk: 8 x columns
        int per, nK, c0, ncol;  // chunks per atom, K values in all (atoms padded to 8)
    } src;
    int nst, nmma, nt;
    WsItem1 item;
    const WsRun* runs;
    const int* grp_t;
    const unsigned char* planes;

    // B producers: `at` = the source slot and chunk of a K value
    struct At {
        int slot, c;
    };
    __device__ __forceinline__ At start(int k) const {
        const int kc = k >> 3, sl = kc / src.per;
        return {sl, kc - sl * src.per};
    }
    __device__ __forceinline__ void advance(At& a, int by) const {
        a.c += by >> 3;
        while (a.c >= src.per) {
            a.c -= src.per;
            ++a.slot;
        }
    }
    __device__ __forceinline__ void load_b(const At& at, int col, int k, float2 (&v)[8]) const {
        if (col >= src.ncol || k >= src.nK) {
            zero8(v);
            return;
        }
        load8(src.x8 + ((int64_t)src.S[at.slot] * src.per + at.c) * src.ldx + 8 * (src.c0 + col), v);
    }
    // lane's copies: one run of groups; MT = 1 takes two K units per stage, the
    // runs of the second on the upper half of the warp
    template <int MT>
    __device__ __forceinline__ WsCopy copy(int lane, uint32_t& total) const {
        const int units = WsGeom<MT>::KSTEPS;
        const int n = item.nrun[0] + (MT == 2 ? item.nrun[1] : 0);
        total = (uint32_t)units * 1024u * (item.ngrp[0] + (MT == 2 ? item.ngrp[1] : 0));
        const int u = MT == 1 ? lane >> 4 : 0, r = MT == 1 ? lane & 15 : lane;
        if (r >= n) return {nullptr, 0, 0, 0};
        const WsRun R = runs[item.run0 + r];
        const int m = r < item.nrun[0] ? 0 : 1;
        return {planes + ((int64_t)R.unit + (int64_t)u * R.step) * 1024, (int64_t)units * R.step * 1024,
                (uint32_t)(m + u) * kUnit + (uint32_t)R.g0 * 1024u, (uint32_t)R.ng * 1024u};
    }
    template <int MT> __device__ __forceinline__ int next_idx(int, int) const { return 0; }
    // (the last stage of MT = 1 may lack its second unit: it repeats the first, against zero B values)
    template <int MT>
    __device__ __forceinline__ void issue(const WsCopy& c, int lane, int st, int, uint32_t dst, uint32_t mb) const {
        if (!c.bytes) return;
        const unsigned char* s = c.src + st * c.step;
        if (MT == 1 && lane >= 16 && 32 * st + 16 >= src.nK) s -= c.step / 2;
        bulk_copy(dst + c.dst, s, c.bytes, mb);
    }
    __device__ __forceinline__ bool valid(int m, int r) const { return (r >> 3) < item.ngrp[m]; }
    __device__ __forceinline__ int64_t dest(int m, int r, int64_t ldt) const {
        return grp_t[item.grp0 + (m ? 16 : 0) + (r >> 3)] * ldt + (r & 7);
    }
};

template <int MT, class Role>
__device__ void ws_tiles(const WsArgs1& a, int it0, int it1, volatile int* abort, Role&& role) {
    for (int it = it0; it < it1 && !*abort; ++it) {
        const WsItem1 item = a.items[it];
        const FarBlockDev B = a.blocks[item.rep];
        const int2 cr = a.colr ? a.colr[item.prob] : make_int2(0, a.nrhs);
        for (int c0 = cr.x; c0 < cr.y && !*abort; c0 += kN) {
            const int nK = 8 * a.per * B.ns;
            WsTile1 T{{a.batoms + B.s_off, a.x8, a.ldx, a.per, nK, c0, min(kN, cr.y - c0)},
                      (nK + WsGeom<MT>::KS - 1) / WsGeom<MT>::KS, 0, MT == 2 && item.ngrp[1] > 0 ? 2 : 1,
                      item, a.runs, a.grp_t, a.planes};
            T.nmma = max(16, (T.src.ncol + 15) / 16 * 16);
            if (!role(T, c0)) return;
        }
    }
}

struct WsTile2 {
    struct Src {
        const int* tidx;  // per chunk of 8 K values: its place in t
        const float2* t;
        int64_t ldt;
        int nK, c0, ncol;
    } src;
    int nst, nmma, nt;
    WsItem2 item;
    const int* qidx;  // per chunk: its 8 KB of planes in a row tile's region
    const unsigned char* planes;
    int64_t rt_bytes, rb;

    // B producers: `at` = the chunk's eight entries of t
    struct At {
        int k, t;
    };
    __device__ __forceinline__ At start(int k) const { return {k, k < src.nK ? src.tidx[k >> 3] : 0}; }
    __device__ __forceinline__ void advance(At& a, int by) const { a = start(a.k + by); }
    __device__ __forceinline__ void load_b(const At& at, int col, int k, float2 (&v)[8]) const {
        if (col >= src.ncol || k >= src.nK) {
            zero8(v);
            return;
        }
        load8(src.t + (int64_t)at.t * src.ldt + 8 * (src.c0 + col), v);
    }
    // lanes 0..3: MT = 2: chunk lane & 1 of row tile lane >> 1; MT = 1: chunk lane.
    // Chunks that follow each other in memory go as one copy, by the first one's lane.
    template <int MT>
    __device__ __forceinline__ WsCopy copy(int lane, uint32_t& total) const {
        const int n = MT == 2 ? 2 * nt : 4;
        total = 8192u * n;
        return {planes + ((int64_t)item.rt + (MT == 2 ? lane >> 1 & 1 : 0)) * rt_bytes, 0, (uint32_t)lane * 8192u,
                lane < n ? 8192u : 0u};
    }
    // the lane's chunk of a stage (read a stage ahead; past the end: the last one, against zero B values)
    template <int MT>
    __device__ __forceinline__ int next_idx(int lane, int st) const {
        return qidx[min(MT == 2 ? 2 * st + (lane & 1) : 4 * st + (lane & 3), (src.nK >> 3) - 1)];
    }
    template <int MT>
    __device__ __forceinline__ void issue(const WsCopy& c, int lane, int, int idx, uint32_t dst, uint32_t mb) const {
        constexpr int W = MT == 2 ? 2 : 4;  // chunks of a stage and row tile
        const int prev = __shfl_up_sync(0xffffffffu, idx, 1);
        const bool first = (lane & (W - 1)) == 0 || idx != prev + 1;
        const unsigned starts = __ballot_sync(0xffffffffu, first) >> lane >> 1;  // later lanes that start a copy
        const int room = W - (lane & (W - 1)), len = min(room, starts ? __ffs(starts) : room);
        if (c.bytes && first) bulk_copy(dst + c.dst, c.src + (int64_t)idx * 8192, 8192u * len, mb);
    }
    __device__ __forceinline__ bool valid(int m, int r) const { return r < item.rows[m]; }
    __device__ __forceinline__ int64_t dest(int m, int r, int64_t) const { return rb + m * kM + r; }
};

template <int MT, class Role>
__device__ void ws_tiles(const WsArgs2& a, int it0, int it1, volatile int* abort, Role&& role) {
    for (int it = it0; it < it1 && !*abort; ++it) {
        const WsItem2 item = a.items[it];
        const int kb = a.kptr[item.atom], nK = 8 * (a.kptr[item.atom + 1] - kb);
        const int2 cr = a.colr ? a.colr[item.prob] : make_int2(0, a.nrhs);
        for (int c0 = cr.x; c0 < cr.y && !*abort; c0 += kN) {
            WsTile2 T{{a.tidx + kb, a.t, a.ldt, nK, c0, min(kN, cr.y - c0)},
                      (nK + WsGeom<MT>::KS - 1) / WsGeom<MT>::KS, 0, MT == 2 && item.rows[1] > 0 ? 2 : 1,
                      item, a.qidx + kb, a.planes, a.rt_bytes, (int64_t)item.atom * a.np + (int64_t)item.rt * kM};
            T.nmma = max(16, (T.src.ncol + 15) / 16 * 16);
            if (!role(T, c0)) return;
        }
    }
}

__device__ void ws_setup(WsCtl& ctl, uint32_t ns) {
    if (threadIdx.x == 0) {
        for (uint32_t i = 0; i < ns; ++i) {
            mbar_init_n(smem_u32(&ctl.full_a[i]), 1);
            mbar_init_n(smem_u32(&ctl.full_b[i]), 2);
            mbar_init_n(smem_u32(&ctl.empty[i]), 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init_n(smem_u32(&ctl.acc_full[i]), 1);
            mbar_init_n(smem_u32(&ctl.acc_empty[i]), 4);
        }
        ctl.abort = 0;
        ctl.g_tma = 0;
        ctl.g_mma = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if ((threadIdx.x >> 5) == kWsWarpMma) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl.tmem)),
                     "r"(kWsTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
}

// wait for what is still in flight (started copies, issued MMAs), free the
// tensor memory, report an abort
__device__ void ws_teardown(WsCtl& ctl, uint32_t ns, int* err) {
    __syncthreads();
    if (threadIdx.x == kWsWarpTma * 32) {
        for (uint32_t g = ctl.g_mma; g < ctl.g_tma; ++g)
            mbar_wait_lim(smem_u32(&ctl.full_a[g % ns]), (g / ns) & 1, kWaitCycles);
    }
    if (threadIdx.x == kWsWarpMma * 32 && ctl.g_mma > 0) {  // the last issued stage's commit
        const uint32_t g = ctl.g_mma - 1;
        mbar_wait_lim(smem_u32(&ctl.empty[g % ns]), (g / ns) & 1, kWaitCycles);
    }
    if (threadIdx.x == 0 && ctl.abort) atomicExch(err, 1);
    fence_before();
    __syncthreads();
    fence_after();
    if ((threadIdx.x >> 5) == kWsWarpMma)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(ctl.tmem), "r"(kWsTmemCols)
                     : "memory");
}

// The B operand of a tile's stages st, st + groups, ...: a thread's NS segments of
// 8 values (neighbouring threads take neighbouring columns of one K chunk, so
// their 16-byte stores fill whole shared-memory wavefronts), read one stage
// ahead and before the wait for the slot, then split and stored.
// Returns the first stage not done, -1 on an abort.
struct ProduceArgs {
    int gtid, groups;
    long long lim;
};
template <int MT, int NS, class TileT>
__device__ __forceinline__ int ws_produce(WsCtl& ctl, const WsRing& ring, const TileT& T, RingPos& p,
                                          const ProduceArgs& a, int st) {
    using G = WsGeom<MT>;
    const int nm = T.nmma, nseg = nm * G::KQ, lane = threadIdx.x & 31;
    int col[NS], kq[NS];
    typename TileT::At at[NS];
#pragma unroll
    for (int u = 0; u < NS; ++u) {
        const int seg = a.gtid + 64 * u;
        kq[u] = seg / nm;
        col[u] = seg < nseg ? seg - kq[u] * nm : -1;
        at[u] = T.start(st * G::KS + 8 * kq[u]);
    }
    float2 vb[NS][8];
    auto load = [&](int s) {
#pragma unroll
        for (int u = 0; u < NS; ++u)
            if (col[u] >= 0) {
                T.load_b(at[u], col[u], s * G::KS + 8 * kq[u], vb[u]);
                T.advance(at[u], a.groups * G::KS);
            }
    };
    load(st);
    for (; st < T.nst; st += a.groups) {
        Chunks cur[NS];
#pragma unroll
        for (int u = 0; u < NS; ++u)
            if (col[u] >= 0) cur[u] = split8(vb[u]);
        if (st + a.groups < T.nst) load(st + a.groups);
        int ok = 1;
        if (lane == 0) ok = ws_wait(ctl, ctl.empty[p.slot], p.par ^ 1, a.lim);
        if (!__shfl_sync(0xffffffffu, ok, 0)) return -1;
        uint4* b0 = ring.b(p.slot, 0);
        uint4* b1 = ring.b(p.slot, 1);
#pragma unroll
        for (int u = 0; u < NS; ++u)
            if (col[u] >= 0) put8_ws(b0, b1, nm, col[u], kq[u], cur[u]);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&ctl.full_b[p.slot]));
        p.step((uint32_t)a.groups, ring.ns);
    }
    return st;
}

// The roles over one phase's tiles.  enumerate: a callable enumerating the
// CTA's tiles; out + dest(m, r) + c (8 in phase 1, ldo in phase 2): where row r of M
// tile m, column c goes.
template <int MT, int PHASE, class TileT, class Enum>
__device__ void ws_run(WsCtl& ctl, const WsRing& ring, int nmax, long long lim, float2* out, int64_t ldo,
                       Enum&& enumerate) {
    using G = WsGeom<MT>;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t accs = 4u * nmax;  // columns of one accumulator
    const uint32_t nbuf = (uint32_t)G::nbuf(nmax);
    if (warp == kWsWarpTma) {
        // ---- A copies: a lane per copy of the stage
        RingPos p;
        uint32_t g = 0;
        enumerate([&](const TileT& T, int) -> bool {
            if (T.nst == 0) return true;
            uint32_t total;
            const WsCopy c = T.template copy<MT>(lane, total);
            int idx = T.template next_idx<MT>(lane, 0);
            for (int st = 0; st < T.nst; ++st, ++g) {
                const int cur = idx;
                if (st + 1 < T.nst) idx = T.template next_idx<MT>(lane, st + 1);
                const uint32_t mb = smem_u32(&ctl.full_a[p.slot]);
                int go = 1;
                if (lane == 0) {
                    go = ws_wait(ctl, ctl.empty[p.slot], p.par ^ 1, lim);  // (passes on the ring's first pass)
                    if (go) mbar_expect_tx(mb, total);
                }
                if (!__shfl_sync(0xffffffffu, go, 0)) return false;
                T.template issue<MT>(c, lane, st, cur, ring.a(p.slot), mb);
                __syncwarp();
                if (lane == 0) ctl.g_tma = g + 1;
                p.step(1, ring.ns);
            }
            return true;
        });
        __syncwarp();
    } else if (warp >= kWsWarpB0 && warp < kWsWarpMma) {
        // ---- B operands: group q (two warps, 64 threads) takes the stages
        // g = q mod G and fills ring slot g mod ns, G = min(4, ns) groups.  It
        // loads a stage's values into registers before it waits for the slot,
        // so the gather from L2 overlaps the MMAs that still read the slot.
        // G <= ns keeps every wait on a slot's "empty" barrier within one
        // phase of it: the group's previous stage g - G waited for the MMAs of
        // stage g - G - ns >= g - 2 ns, so the phase of stage g - ns that this
        // wait asks for is the barrier's current or last completed one, never
        // one that a parity test would confuse with an older phase.
        const int q = (warp - kWsWarpB0) >> 1;
        const int gtid = tid - (kWsWarpB0 + 2 * q) * 32;
        const uint32_t ngroups = ring.ns < (uint32_t)kWsGroups ? ring.ns : (uint32_t)kWsGroups;
        RingPos p;
        p.step((uint32_t)q, ring.ns);
        int wait = q;  // stages until this group's next one
        if ((uint32_t)q < ngroups) enumerate([&](const TileT& T, int) -> bool {
            if (wait >= T.nst) {
                wait -= T.nst;
                return true;
            }
            const int nseg = T.nmma * G::KQ;  // segments of 8 values, 64 threads
            const ProduceArgs pa{gtid, (int)ngroups, lim};
            const int st = nseg <= 64 ? ws_produce<MT, 1>(ctl, ring, T, p, pa, wait)
                                      : ws_produce<MT, 2>(ctl, ring, T, p, pa, wait);
            if (st < 0) return false;
            wait = st - T.nst;
            return true;
        });
    } else if (warp == kWsWarpMma) {
        // ---- MMA issuer: the warp runs the loop together, so that the operands stay
        // in uniform registers; one elected lane issues
        const bool leader = elect_one();
        RingPos p, ab;  // stage ring, accumulator buffers
        uint32_t g = 0;
        const uint32_t a0 = ring.a(0) >> 4, dslot = ring.stride >> 4, dstack = ring.bstack;
        enumerate([&](const TileT& T, int) -> bool {
            if (T.nst == 0) return true;
            if (!ws_wait_warp(ctl, ctl.acc_empty[ab.slot], ab.par ^ 1, lim)) return false;
            const uint32_t tm = ctl.tmem + ab.slot * MT * accs;
            const uint32_t id4 = idesc(4 * T.nmma, false), id2 = idesc(2 * T.nmma, false);
            const uint32_t lbob = (uint32_t)(4 * T.nmma * 16), lb = (lbob >> 4) << 16, kb = 2 * lbob >> 4;
            const int nt = MT == 2 ? T.nt : 1;
            uint32_t acc0 = 0;
            for (int st = 0; st < T.nst; ++st, ++g) {
                if (!ws_wait_warp(ctl, ctl.full_a[p.slot], p.par, lim) ||
                    !ws_wait_warp(ctl, ctl.full_b[p.slot], p.par, lim))
                    return false;
                fence_after();
                const uint32_t a = a0 + p.slot * dslot, b0 = a + (2 * kUnit >> 4) + lb, b1 = b0 + dstack;
                if (leader) {
                    mma_kstep_ws<PHASE>(a, b0, b1, tm, id4, id2, acc0);
                    if (MT == 1) mma_kstep_ws<PHASE>(a + (kUnit >> 4), b0 + kb, b1 + kb, tm, id4, id2, 1u);
                    else if (nt == 2) mma_kstep_ws<PHASE>(a + (kUnit >> 4), b0, b1, tm + accs, id4, id2, acc0);
                    umma_commit(smem_u32(&ctl.empty[p.slot]));
                    ctl.g_mma = g + 1;
                }
                __syncwarp();
                acc0 = 1;
                p.step(1, ring.ns);
            }
            if (leader) umma_commit(smem_u32(&ctl.acc_full[ab.slot]));
            __syncwarp();
            ab.step(1, nbuf);
            return true;
        });
    } else {
        // ---- epilogue (warps 0-3, tensor-memory lane quarter = warp)
        RingPos ab;
        const int r = warp * 32 + lane;
        const uint32_t lane_base = (uint32_t)(warp * 32) << 16;
        enumerate([&](const TileT& T, int c0) -> bool {
            const int ncol = T.src.ncol;
            if (T.nst == 0) {
                for (int m = 0; m < T.nt; ++m)  // (phase 2: an atom without far blocks)
                    if (T.valid(m, r))
                        for (int c = 0; c < ncol; ++c)
                            out[T.dest(m, r, ldo) + (int64_t)(c0 + c) * (PHASE == 1 ? 8 : ldo)] = make_float2(0.f, 0.f);
                return true;
            }
            int ok = 1;
            if (lane == 0) ok = ws_wait(ctl, ctl.acc_full[ab.slot], ab.par, lim);
            if (!__shfl_sync(0xffffffffu, ok, 0)) return false;
            fence_after();
            const int nm = T.nmma;
            for (int m = 0; m < T.nt; ++m) {
                const uint32_t base = ctl.tmem + (ab.slot * MT + m) * accs + lane_base;
                const bool mine = T.valid(m, r);
                float2* o = out + (mine ? T.dest(m, r, ldo) : 0) + (int64_t)c0 * (PHASE == 1 ? 8 : ldo);
                for (int cb = 0; cb < ncol; cb += 16) {
                    float ra[16], ia[16], rb[16], ib[16];
                    tmem_ld16(base + cb, ra);
                    tmem_ld16(base + nm + cb, ia);
                    tmem_ld16(base + 2 * nm + cb, rb);
                    tmem_ld16(base + 3 * nm + cb, ib);
                    tmem_wait_ld();
                    if (mine) {
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            if (cb + i < ncol)
                                o[(int64_t)(cb + i) * (PHASE == 1 ? 8 : ldo)] = make_float2(ra[i] + rb[i], ia[i] + ib[i]);
                    }
                }
            }
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&ctl.acc_empty[ab.slot]));
            ab.step(1, nbuf);
            return true;
        });
    }
}

template <int MT, int PHASE, class TileT, class Args>
__device__ __forceinline__ void ws_body(const Args& a, float2* out, int64_t ldo, int nmax, int* err, long long lim) {
    extern __shared__ __align__(1024) unsigned char smem[];
    const WsRing ring = ws_ring<MT>(smem, nmax);
    __shared__ WsCtl ctl;
    ws_setup(ctl, ring.ns);
    const int it0 = a.cta_ptr[blockIdx.x], it1 = a.cta_ptr[blockIdx.x + 1];
    ws_run<MT, PHASE, TileT>(ctl, ring, nmax, lim, out, ldo,
                             [&](auto&& role) { ws_tiles<MT>(a, it0, it1, &ctl.abort, role); });
    ws_teardown(ctl, ring.ns, err);
}
template <int MT>
__global__ void __launch_bounds__(kWsThr, 1) u1w_kernel(WsArgs1 a, float2* t, int64_t ldt, int nmax, int* err,
                                                         long long lim) {
    ws_body<MT, 1, WsTile1>(a, t, ldt, nmax, err, lim);
}
template <int MT>
__global__ void __launch_bounds__(kWsThr, 1) u2w_kernel(WsArgs2 a, float2* F, int64_t ldf, int nmax, int* err,
                                                         long long lim) {
    ws_body<MT, 2, WsTile2>(a, F, ldf, nmax, err, lim);
}

// ---- packing: a factor storage's planes, once ---------------------------------
// R: thread = one 8-value K chunk of one row; consecutive threads take the 8 rows
// of a group, then the two chunks of a unit
__global__ void __launch_bounds__(256) k_pack_r(const WsClass* __restrict__ cls, int ncls, int64_t total, int np,
                                                int per, const float2* __restrict__ fac,
                                                unsigned char* __restrict__ planes) {
    for (int64_t w = (int64_t)blockIdx.x * 256 + threadIdx.x; w < total; w += (int64_t)gridDim.x * 256) {
        const int64_t unit = w >> 4;  // kilobyte: (K unit, group)
        int lo = 0, hi = ncls - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (cls[mid].r_unit <= unit) lo = mid;
            else hi = mid - 1;
        }
        const WsClass c = cls[lo];
        const int G = (c.rank + 7) / 8;
        const int64_t u = unit - c.r_unit;
        const int ku = (int)(u / G), g = (int)(u - (int64_t)ku * G), row = g * 8 + (int)(w & 7), q = (int)(w >> 3) & 1;
        const int kc = ku * 2 + q, slot = kc / per, o = (kc - slot * per) * 8;  // chunk of an atom padded to 8
        float2 v[8];
        const float2* src = fac + c.rh_off + (int64_t)row * c.n + slot * np + o;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const float2 x = row < c.rank && slot * np < c.n && o + e < np ? __ldg(src + e) : make_float2(0.f, 0.f);
            v[e] = make_float2(x.x, -x.y);
        }
        const Chunks p = split8(v);
        uint4* out = reinterpret_cast<uint4*>(planes + unit * 1024) + q * 8 + (w & 7);
        out[0] = p.rh;
        out[16] = p.rl;
        out[32] = p.ih;
        out[48] = p.il;
    }
}

// x as [chunk of an atom (8 values, zero padded)][column][8]: the 64 columns of a
// chunk in a row, read by every tile whose source box holds the atom.  Thread =
// one chunk of one column; neighbouring threads take neighbouring chunks.
__global__ void __launch_bounds__(256) k_x8(const float2* __restrict__ x, int64_t ldx, int np, int per, int64_t chunks,
                                            int nrhs, float2* __restrict__ out) {
    for (int64_t w = (int64_t)blockIdx.x * 256 + threadIdx.x; w < chunks; w += (int64_t)gridDim.x * 256) {
        const int64_t atom = w / per;
        const int c = (int)(w - atom * per), col = blockIdx.y;
        const float4* src = reinterpret_cast<const float4*>(x + col * ldx + atom * np + 8 * c);
        float4* dst = reinterpret_cast<float4*>(out + (w * nrhs + col) * 8);
#pragma unroll
        for (int e = 0; e < 4; ++e)  // np is even
            dst[e] = 8 * c + 2 * e < np ? __ldg(src + e) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// Q: thread = one row of a chunk of 8 K values
__global__ void __launch_bounds__(128) k_pack_q(const WsClass* __restrict__ cls, int ncls, int64_t total, int np,
                                                int nrt, const float2* __restrict__ fac, unsigned char* __restrict__ planes) {
    for (int64_t w = blockIdx.x; w < total * nrt; w += gridDim.x) {
        const int rt = (int)(w / total);
        const int64_t chunk = w - rt * total;
        int lo = 0, hi = ncls - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (cls[mid].q_chunk <= chunk) lo = mid;
            else hi = mid - 1;
        }
        const WsClass c = cls[lo];
        const int G = (c.rank + 7) / 8;
        const int64_t u = chunk - c.q_chunk;
        const int k8 = (int)(u % G), slot = (int)(u / G);
        const int row = rt * kM + (int)threadIdx.x;
        float2 v[8];
        const float2* src = fac + c.q_off + (int64_t)slot * np + row;
#pragma unroll
        for (int e = 0; e < 8; ++e)
            v[e] = row < np && k8 * 8 + e < c.rank ? __ldg(src + (int64_t)(k8 * 8 + e) * c.m) : make_float2(0.f, 0.f);
        const Chunks p = split8(v);
        uint4* out = reinterpret_cast<uint4*>(planes + w * 8192) + threadIdx.x;
        out[0] = p.rh;
        out[128] = p.rl;
        out[256] = p.ih;
        out[384] = p.il;
    }
}

std::once_flag g_ws_attr_once;

}  // namespace

size_t ws_plane_bytes(const Op& op) {
    return (size_t)op.ws_r_units * 1024 + (size_t)op.ws_q_chunks * ((op.np + kM - 1) / kM) * 8192;
}

bool ws_pack(Op& op, cudaStream_t s) {
    if (op.fprec != VIE_C64) fail(VIE_ERR_INVALID_ARG, "the tcgen05 apply needs VIE_C64 factors");
    std::call_once(g_ws_attr_once, [] {
        cudaFuncSetAttribute(u1w_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kWsSmemBytes);
        cudaFuncSetAttribute(u2w_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kWsSmemBytes);
        cudaFuncSetAttribute(u1w_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, kWsSmemBytes);
        cudaFuncSetAttribute(u2w_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, kWsSmemBytes);
    });
    if (!op.d_err.p) {
        op.d_err.alloc(sizeof(int));
        VIE_CUDA(cudaMemsetAsync(op.d_err.p, 0, sizeof(int), s));
    }
    if (op.ws_packed) return true;
    if (op.ws_pack_failed) return false;
    build_ws_lists(op);
    const size_t b1 = (size_t)op.ws_r_units * 1024, b2 = ws_plane_bytes(op) - b1;
    size_t free_b = 0, total_b = 0;
    VIE_CUDA(cudaMemGetInfo(&free_b, &total_b));
    if (b1 + b2 + ((size_t)1 << 30) > free_b) {  // keep 1 GiB for the solver
        op.ws_pack_failed = true;
        return false;
    }
    op.d_ws_r.alloc(std::max<size_t>(b1, 16));
    op.d_ws_q.alloc(std::max<size_t>(b2, 16));
    if (op.ws_ncls > 0) {
        const int64_t w1 = op.ws_r_units * 16;
        k_pack_r<<<(unsigned)std::min<int64_t>((w1 + 255) / 256, 64ll * op.ctx->n_sm), 256, 0, s>>>(
            op.d_ws_cls.as<WsClass>(), op.ws_ncls, w1, op.np, (op.np + 7) / 8, op.fac<float2>(),
            op.d_ws_r.as<unsigned char>());
        VIE_CHECK_LAUNCH();
        k_pack_q<<<(unsigned)std::min<int64_t>(op.ws_q_chunks, 64ll * op.ctx->n_sm), 128, 0, s>>>(
            op.d_ws_cls.as<WsClass>(), op.ws_ncls, op.ws_q_chunks, op.np, (op.np + kM - 1) / kM, op.fac<float2>(),
            op.d_ws_q.as<unsigned char>());
        VIE_CHECK_LAUNCH();
    }
    op.ws_packed = true;
    return true;
}

void ws_reserve(Op& op, int nrhs) {
    const size_t need = (size_t)std::max<int64_t>(op.ws_t_total, 1) * nrhs * sizeof(float2);
    if (op.d_t.bytes < need) op.d_t.alloc(need);
    const size_t need_x = (size_t)op.N * ((op.np + 7) / 8) * 8 * nrhs * sizeof(float2);
    if (op.d_xs.bytes < need_x) op.d_xs.alloc(need_x);
}

// MT = 1: variant 9 (one row tile per B tile); MT = 2: variant 10 (two)
template <int MT>
static void apply_far_ws(Op& op, const float2* x, int64_t ldx, float2* F, int64_t ldf, int nrhs, cudaStream_t s) {
    if (!ws_pack(op, s)) {  // not enough memory for the planes: the kernel that splits A itself
        apply_far_umma(op, x, ldx, F, ldf, nrhs, s);
        return;
    }
    if (((uintptr_t)x & 15) || (ldx & 1)) fail(VIE_ERR_INVALID_ARG, "tensor-core apply: x must be 16-byte aligned");
    ws_reserve(op, nrhs);
    const long long lim = wait_limit(kWaitCycles);
    const int nc = op.ctx->n_sm;
    // the widest tile: 64 columns, or all of them when fewer (a tile never
    // spans two problems' column ranges, so it is no wider than this either)
    const int nmax = std::max(16, (std::min(nrhs, kN) + 15) / 16 * 16);
    const size_t smem = (size_t)WsGeom<MT>::stages(nmax) * WsGeom<MT>::stride(nmax);
    constexpr int v = MT - 1;
    if (op.n_ws1[v] > 0) {
        const int per = (op.np + 7) / 8;
        const int64_t chunks = (int64_t)op.N * per;
        for (int c0 = 0; c0 < nrhs; c0 += 65535) {
            const dim3 grid((unsigned)std::min<int64_t>((chunks + 255) / 256, 65535), (unsigned)std::min(nrhs - c0, 65535));
            k_x8<<<grid, 256, 0, s>>>(
                x + c0 * ldx, ldx, op.np, per, chunks, nrhs, op.d_xs.as<float2>() + 8 * c0);
            VIE_CHECK_LAUNCH();
        }
        const WsArgs1 a{op.d_blocks.as<FarBlockDev>(), op.d_block_atoms.as<int>(), op.d_ws1_items[v].as<WsItem1>(),
                        op.d_ws1_cta[v].as<int>(), op.d_ws_runs[v].as<WsRun>(), op.d_ws_grp.as<int>(),
                        op.d_ws_r.as<unsigned char>(), op.d_xs.as<float2>(), 8ll * nrhs, per, nrhs, op.colr};
        u1w_kernel<MT><<<nc, kWsThr, smem, s>>>(a, op.d_t.as<float2>(), 8ll * nrhs, nmax, op.d_err.as<int>(), lim);
        VIE_CHECK_LAUNCH();
    }
    const WsArgs2 a{op.d_ws2_items[v].as<WsItem2>(), op.d_ws2_cta[v].as<int>(), op.d_ws_kptr.as<int>(),
                    op.d_ws_qidx.as<int>(), op.d_ws_tidx.as<int>(), op.d_ws_q.as<unsigned char>(),
                    op.d_t.as<float2>(), 8ll * nrhs, (int64_t)op.ws_q_chunks * 8192, op.np, nrhs, op.colr};
    u2w_kernel<MT><<<nc, kWsThr, smem, s>>>(a, F, ldf, nmax, op.d_err.as<int>(), lim);
    VIE_CHECK_LAUNCH();
}

void apply_far_umma_ws(Op& op, const float2* x, int64_t ldx, float2* F, int64_t ldf, int nrhs, cudaStream_t s) {
    // wider, a producer thread would hold four segments of B of one 32-K stage: two
    // row tiles per B tile take half of them
    if (nrhs <= 32) apply_far_ws<1>(op, x, ldx, F, ldf, nrhs, s);
    else apply_far_ws<2>(op, x, ldx, F, ldf, nrhs, s);
}

void apply_far_umma_ws2(Op& op, const float2* x, int64_t ldx, float2* F, int64_t ldf, int nrhs, cudaStream_t s) {
    apply_far_ws<2>(op, x, ldx, F, ldf, nrhs, s);
}

}  // namespace vie
