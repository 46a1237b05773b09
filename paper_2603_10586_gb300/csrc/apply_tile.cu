// Far apply F = sum_b Q_b (R_b x) by register tiles, for operators whose far
// blocks share factors or for several right-hand sides (complex float32,
// double-float and complex float64 arithmetic).
//
// Blocks with the same factor storage (translated copies) form a class.  A
// class's members times the right-hand sides are the columns of two plain
// matrix products with the class's factors:
//   phase 1:  t[:, col]  = R x[S_col, rhs]      (rank x n) (n x columns)
//   phase 2:  P[:, col]  = Q t[:, col]          (m x rank) (rank x columns)
//   phase 3:  F_a        = sum of the P rows of atom a, in its entry list's order
// An item is one class, up to kTileMembers of its members and, in phase 1, up
// to 64 rows (fewer on small operators and in complex128, see build_apply_lists)
// and Op::tile_seg columns of R (the segments' partial t are added in
// order where phase 2 reads them, so a long row is neither a long chain nor a
// late CTA), in phase 2 up to 256 rows of Q.  Every output element is written by
// one thread and every sum has a fixed order: the result does not depend on the
// schedule.
//
// What bounds it: the float32 (or float64) pipes, with the shared-memory reads
// close behind.  A warp holds a tile of 64 rows x 16 columns (float32; 8 columns
// otherwise, or when there are no more), 4 x 8 complex accumulators per thread, so
// a K value costs a thread 128 FMAs and 12 shared-memory loads.  The four warps of
// a CTA share out what there is: in phase 1 the columns and, where there are
// few of them, the K range (groups added in order at the end); in phase 2 the
// rows and then the columns.  Operands go through two shared-memory buffers
// by cp.async (the factor, and x gathered over the source atoms); t is small and
// goes through registers.
//
// Measured on one GB300 (fused apply, against the kernels that read a factor once
// per four copies of one right-hand side or once per four right-hand sides):
//   4 x 4 array of 3^3 cubes, 1 column, complex float32       38 -> 32 us
//   16 x 16 array of 6^3 cubes, 1 column, complex float32    953 -> 486 us
//   28 x 28 array of 3^3 cubes, 5 columns, complex float32  4105 -> 1132 us
//   16 x 16 array of 4^3 cubes, 24 columns, double-float    20.9 -> 17.0 ms
//   12 x 12 array of 3^3 cubes, 3 columns, complex float64  3840 -> 2079 us
//    8 x 8 array of 3^3 cubes, 1 column, complex float64     642 -> 400 us
#include <algorithm>
#include <atomic>

#include "common.h"
#include "cplx.cuh"
#include "farmac.cuh"
#include "tilemma.cuh"

namespace vie {

namespace {

constexpr int kThr = 128;    // four warps
template <class TF> constexpr bool kWide = std::is_same<TF, double2>::value;
// rows per tile of phase 1, and per warp of phase 2
template <class TF> constexpr int kTM1 = kWide<TF> ? kTileRows1Wide : kTileRows1;
template <class TF> constexpr int kTM2 = kWide<TF> ? kTileRows2Wide : kTileRows2 / 4;

// Staged operands: A1 [row][K], B [column][K] (K contiguous, as in memory) with
// one 16-byte unit of padding per row, so that threads a row apart read other
// banks and a load takes two float32 K values; A2 [K][row].
// phase 1: WN warps side by side, WK = 4 / WN groups along K
template <class TF, class TX, int WN, int J>
struct Shape1 {
    static constexpr int WK = 4 / WN, TN = 2 * J * WN;
    static constexpr int KC = WN == 4 ? 16 : 32;     // K values per stage
    static constexpr int KG = KC / WK;               // of those, per K group
    static constexpr int LA = KC + kE<TF>, LB = KC + kE<TX>;
    static constexpr size_t a_pad = (size_t)kTM1<TF> * LA * sizeof(TF);
    static constexpr size_t stage = a_pad + (size_t)TN * LB * sizeof(TX);
};
// phase 2: RW warps down the rows, CW = 4 / RW side by side
template <class TF, class TX, int RW, int J>
struct Shape2 {
    static constexpr int CW = 4 / RW, TN = 2 * J * CW, KC = 8;
    static constexpr int LA = kTM2<TF> * RW, LB = KC + kE<TX>;
    static constexpr size_t a_pad = (size_t)KC * LA * sizeof(TF);
    static constexpr size_t stage = a_pad + (size_t)TN * LB * sizeof(TX);
};
// complex128 asks for more than it uses, so that an SM holds two CTAs of phase 1
// and three of phase 2, which keep its float64 units busy, and takes the next
// when one is done (8 x 8 array of 3^3 cubes, 1 column: 575 us with all it can hold, 447 so)
constexpr size_t kWideSmem1 = 84 << 10, kWideSmem2 = 68 << 10;
template <class TF, class TX> constexpr size_t smem_bytes(int phase) {
    constexpr int J = kJ<TX>;
    if (kWide<TF> && phase == 1) return kWideSmem1;
    if (phase == 1)
        return 2 * std::max({Shape1<TF, TX, 4, J>::stage, Shape1<TF, TX, 2, J>::stage, Shape1<TF, TX, 1, J>::stage});
    if (kWide<TF>) return kWideSmem2;
    return 2 * std::max({Shape2<TF, TX, 4, J>::stage, Shape2<TF, TX, 2, J>::stage, Shape2<TF, TX, 1, J>::stage});
}

static_assert(2 * std::max({Shape1<double2, double2, 4, 4>::stage, Shape1<double2, double2, 2, 4>::stage,
                            Shape1<double2, double2, 1, 4>::stage}) <= kWideSmem1 &&
              2 * Shape2<double2, double2, 1, 4>::stage <= kWideSmem2);

struct TileArgs {
    const int* batoms;
    const FarTile* items;
    const FarMember* mem;
    const int2* colr;
    int np, rhs0, nrhs;      // right-hand sides [rhs0, rhs0 + nrhs) of the call in this pass
    int64_t ldx, ldt, ldp;
};

// columns of this item: member j of the group, right-hand side c0 + c
struct Cols {
    int c0, nc, n;  // first right-hand side, their number, columns in all
    float inv;      // 1 / nc
    // column -> (member, right-hand side); exact: columns stay below 2^16
    __device__ __forceinline__ int member(int col) const { return (int)(((float)col + 0.5f) * inv); }
};
__device__ __forceinline__ Cols cols_of(const TileArgs& a, const FarTile& it) {
    int lo = a.rhs0, hi = a.rhs0 + a.nrhs;
    if (a.colr) {
        const int2 r = a.colr[it.prob];
        lo = max(lo, r.x);
        hi = min(hi, r.y);
    }
    const int nc = max(0, hi - lo);
    return {lo, nc, nc * it.nm, 1.f / (float)max(nc, 1)};
}

// ---------------------------------------------------------------------------
// phase 1, columns [q0, q0 + TN) of the item
// ---------------------------------------------------------------------------
template <class TF, class TX, int WN, int J, int RA>
__device__ void tile1(unsigned char* smem, const TileArgs& a, const FarTile& it, const Cols& C, int q0,
                      const TF* __restrict__ fac, const TX* __restrict__ x, TX* __restrict__ t) {
    using S = Shape1<TF, TX, WN, J>;
    using TA = typename AccOf<TX>::t;
    constexpr int EA = kE<TF>, EB = kE<TX>;
    constexpr int UA = S::KC / EA, UB = S::KC / EB;  // 16-byte units per staged row and column
    constexpr int RA_ = kThr / UA, RB = kThr / UB;   // rows and columns staged at a time
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int wn = warp % WN, wk = warp / WN, tr = lane & 15, tc = lane >> 4;
    const int ka = tid % UA * EA, pa = tid / UA, kb = tid % UB * EB, pb = tid / UB;
    const FarMember* mem = a.mem + it.first;
    const int nst = (it.k1 - it.k0 + S::KC - 1) / S::KC;
    const TF* RH = fac + it.off + (int64_t)(it.row0 + pa) * it.ld + it.k0 + ka;
    const int64_t rstep = (int64_t)RA_ * it.ld;
    // the columns that this thread stages: pb, pb + RB, ...
    constexpr int NB = (S::TN + RB - 1) / RB;
    const TX* xc[NB];
    const int* Sc[NB];
    unsigned live = 0;
#pragma unroll
    for (int u = 0; u < NB; ++u) {
        const int q = pb + u * RB, col = q0 + q;
        const bool ok = q < S::TN && col < C.n;
        const int j = ok ? C.member(col) : 0, c = ok ? col - j * C.nc : 0;
        xc[u] = x + (int64_t)(C.c0 + c) * a.ldx;
        Sc[u] = a.batoms + mem[j].s_off;
        live |= ok ? 1u << u : 0u;
    }
    // (k1, the atoms' sizes and the segments are even, so a unit never straddles)
    int kpos = it.k0 + kb, slot = kpos / a.np, off = kpos - slot * a.np, kf = it.k0 + ka;
    const TX* xs[NB];  // this thread's K values in the column's current atom
    auto enter_slot = [&] {
#pragma unroll
        for (int u = 0; u < NB; ++u) xs[u] = kpos < it.k1 ? xc[u] + (int64_t)Sc[u][slot] * a.np + off : x;
    };
    enter_slot();
    auto fill = [&](int s) {
        unsigned char* st = smem + (s & 1) * S::stage;
        TF* As = reinterpret_cast<TF*>(st) + pa * S::LA + ka;
        TX* Bs = reinterpret_cast<TX*>(st + S::a_pad) + pb * S::LB + kb;
        const TF* src = RH;
#pragma unroll
        for (int r = 0; r < 16 * RA; r += RA_) {
            if (RA_ <= 16 * RA || pa < 16 * RA) {
                const bool ok = kf < it.k1 && r + pa < it.rows;
                cp_async16(As + r * S::LA, ok ? src : fac, ok);
            }
            src += rstep;
        }
        const bool kin = kpos < it.k1;
#pragma unroll
        for (int u = 0; u < NB; ++u)
            if (pb + u * RB < S::TN) {
                const bool ok = kin && ((live >> u) & 1);
                cp_async16(Bs + u * RB * S::LB, ok ? xs[u] : x, ok);
            }
        cp_commit();
        RH += S::KC;
        kf += S::KC;
        kpos += S::KC;
        off += S::KC;
        if (off < a.np) {
#pragma unroll
            for (int u = 0; u < NB; ++u) xs[u] += S::KC;
        } else {
            while (off >= a.np) { off -= a.np; ++slot; }
            enter_slot();
        }
    };
    TA acc[RA][J];
    zero_acc(acc);
    fill(0);
    for (int s = 0; s < nst; ++s) {
        if (s + 1 < nst) {
            fill(s + 1);
            cp_wait<1>();
        } else {
            cp_wait<0>();
        }
        __syncthreads();
        const unsigned char* st = smem + (s & 1) * S::stage;
        mma_stage<TF, TX, TA, 1, S::KG, S::LA, S::LB, RA, J>(
            reinterpret_cast<const TF*>(st) + tr * S::LA + wk * S::KG,
            reinterpret_cast<const TX*>(st + S::a_pad) + (wn * 2 * J + tc) * S::LB + wk * S::KG, acc);
        __syncthreads();
    }
    if (S::WK > 1) {  // the K groups' sums added in order
        TA* buf = reinterpret_cast<TA*>(smem);  // [warp column][i][j][lane], one group at a time
#pragma unroll
        for (int g = 1; g < S::WK; ++g) {
            if (wk == g)
#pragma unroll
                for (int i = 0; i < RA; ++i)
#pragma unroll
                    for (int j = 0; j < J; ++j) buf[((wn * RA + i) * J + j) * 32 + lane] = acc[i][j];
            __syncthreads();
            if (wk == 0)
#pragma unroll
                for (int i = 0; i < RA; ++i)
#pragma unroll
                    for (int j = 0; j < J; ++j) acc_add(acc[i][j], buf[((wn * RA + i) * J + j) * 32 + lane]);
            __syncthreads();
        }
    }
    if (wk == 0)
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const int col = q0 + wn * 2 * J + tc + 2 * j;
            if (col < C.n) {
                const int m = C.member(col), c = col - m * C.nc;
                TX* out = t + mem[m].toff + (int64_t)it.seg * it.rank + it.row0 + (int64_t)(C.c0 + c - a.rhs0) * a.ldt;
#pragma unroll
                for (int i = 0; i < RA; ++i)
                    if (tr + 16 * i < it.rows) store(out + tr + 16 * i, acc[i][j]);
            }
        }
}

// ---------------------------------------------------------------------------
// phase 2, columns [q0, q0 + TN) of the item; warp row wr takes rows
// [wr pw, wr pw + pw) of it, in a thread two neighbouring rows (float32) at a time
// ---------------------------------------------------------------------------
__device__ __forceinline__ int warp_rows(int rows, int RW) { return ((rows + RW - 1) / RW + 1) / 2 * 2; }

template <class TF, class TX, int RW, int J, int RA>
__device__ void tile2(unsigned char* smem, const TileArgs& a, const FarTile& it, const Cols& C, int q0,
                      const TF* __restrict__ fac, const TX* __restrict__ t, TX* __restrict__ P) {
    using S = Shape2<TF, TX, RW, J>;
    using TA = typename AccOf<TX>::t;
    constexpr int KR = kThr / S::KC;  // columns of t staged at a time
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int wr = warp % RW, wc = warp / RW, tr = lane & 15, tc = lane >> 4;
    const int kk = tid % S::KC, part = tid / S::KC;
    const FarMember* mem = a.mem + it.first;
    const int K = it.rank, nst = (K + S::KC - 1) / S::KC;
    constexpr int EA = kE<TF>;
    const int pw = warp_rows(it.rows, RW);
    // factor: units of EA rows, LA / EA of them per K value, KA K values at a time
    // (a tile of 256 rows x 8 bytes is exactly one K value of the CTA)
    constexpr int UR = S::LA / EA, KA = kThr / UR > 0 ? kThr / UR : 1, NU = (UR + kThr - 1) / kThr;
    const int ur = (tid % UR) * EA, uk = tid / UR;
    const TF* Q = fac + it.off + it.row0 + ur + (int64_t)uk * it.ld;
    auto fill_a = [&](int s) {
        TF* As = reinterpret_cast<TF*>(smem + (s & 1) * S::stage) + uk * S::LA + ur;
        const TF* src = Q + (int64_t)s * S::KC * it.ld;
#pragma unroll
        for (int k = 0; k < S::KC; k += KA) {
#pragma unroll
            for (int h = 0; h < NU; ++h) {
                const bool ok = s * S::KC + k + uk < K && ur + h * kThr * EA < it.rows;
                cp_async16(As + k * S::LA + h * kThr * EA, ok ? src + h * kThr * EA : fac, ok);
            }
            src += (int64_t)KA * it.ld;
        }
        cp_commit();
    };
    constexpr int NB = (S::TN + KR - 1) / KR;
    const TX* tb[NB];
    unsigned live = 0;
#pragma unroll
    for (int u = 0; u < NB; ++u) {
        const int q = part + u * KR, col = q0 + q;
        const bool ok = q < S::TN && col < C.n;
        const int j = ok ? C.member(col) : 0, c = ok ? col - j * C.nc : 0;
        tb[u] = t + mem[j].toff + (int64_t)(C.c0 + c - a.rhs0) * a.ldt + kk;
        live |= ok ? 1u << u : 0u;
    }
    TX bv[NB];
    auto load_b = [&](int s) {
        const bool kin = s * S::KC + kk < K;
#pragma unroll
        for (int u = 0; u < NB; ++u) bv[u] = kin && ((live >> u) & 1) ? tb[u][s * S::KC] : TX{};
    };
    auto store_b = [&](int s) {
        TX* Bs = reinterpret_cast<TX*>(smem + (s & 1) * S::stage + S::a_pad) + part * S::LB + kk;
#pragma unroll
        for (int u = 0; u < NB; ++u)
            if (part + u * KR < S::TN) Bs[u * KR * S::LB] = bv[u];
    };
    TA acc[RA][J];
    zero_acc(acc);
    const int rows = min(pw, it.rows - wr * pw);          // (none for a warp past the last row)
    const bool busy = rows > 0 && q0 + wc * 2 * J < C.n;  // (nor past the last column)
    fill_a(0);
    load_b(0);
    for (int s = 0; s < nst; ++s) {
        store_b(s);
        if (s + 1 < nst) {
            fill_a(s + 1);
            load_b(s + 1);
            cp_wait<1>();
        } else {
            cp_wait<0>();
        }
        __syncthreads();
        const unsigned char* st = smem + (s & 1) * S::stage;
        if (busy) mma_stage<TF, TX, TA, 2, S::KC, S::LA, S::LB, RA, J>(
            reinterpret_cast<const TF*>(st) + wr * pw + EA * tr,
            reinterpret_cast<const TX*>(st + S::a_pad) + (wc * 2 * J + tc) * S::LB, acc);
        __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < J; ++j) {
        const int col = q0 + wc * 2 * J + tc + 2 * j;
        if (col < C.n) {
            const int m = C.member(col), c = col - m * C.nc;
            TX* out = P + mem[m].poff + it.row0 + wr * pw + (int64_t)(C.c0 + c - a.rhs0) * a.ldp;
#pragma unroll
            for (int i = 0; i < RA; ++i) {
                const int r = EA == 2 ? 32 * (i >> 1) + 2 * tr + (i & 1) : 16 * i + tr;
                if (r < rows) store(out + r, acc[i][j]);
            }
        }
    }
}

template <class TF, class TX, int PHASE, int W, int J>
__device__ __forceinline__ void tile_rows(unsigned char* smem, const TileArgs& a, const FarTile& it,
                                          const Cols& C, int q0, const TF* fac, const TX* in,
                                          TX* out) {
    const int r = PHASE == 1 ? it.rows : warp_rows(it.rows, W);  // rows of a warp tile
    if constexpr (PHASE == 1 && kWide<TF>) {
        tile1<TF, TX, W, J, 1>(smem, a, it, C, q0, fac, in, out);
    } else if constexpr (PHASE == 1) {
        if (r > 48) tile1<TF, TX, W, J, 4>(smem, a, it, C, q0, fac, in, out);
        else if (r > 32) tile1<TF, TX, W, J, 3>(smem, a, it, C, q0, fac, in, out);
        else if (r > 16 || kE<TX> > 1) tile1<TF, TX, W, J, 2>(smem, a, it, C, q0, fac, in, out);
        else if constexpr (kE<TX> == 1) tile1<TF, TX, W, J, 1>(smem, a, it, C, q0, fac, in, out);
    } else if constexpr (kWide<TF>) {
        if (r > 16) tile2<TF, TX, W, J, 2>(smem, a, it, C, q0, fac, in, out);
        else tile2<TF, TX, W, J, 1>(smem, a, it, C, q0, fac, in, out);
    } else {
        if (r > 32) tile2<TF, TX, W, J, 4>(smem, a, it, C, q0, fac, in, out);
        else tile2<TF, TX, W, J, 2>(smem, a, it, C, q0, fac, in, out);
    }
}

// blockIdx.x: item; its column tiles are dealt out along blockIdx.y
template <class TF, class TX, int PHASE>
__global__ void __launch_bounds__(kThr, std::is_same<TX, float4>::value ? 4 : 3)
k_tile(TileArgs a, const TF* __restrict__ fac, const TX* __restrict__ in, TX* __restrict__ out) {
    extern __shared__ __align__(16) unsigned char tile_smem[];
    constexpr int J = kJ<TX>, H = J / 2;  // columns per thread: full, and for the last few
    const FarTile it = a.items[blockIdx.x];
    const Cols C = cols_of(a, it);
    if constexpr (PHASE == 1) {
        for (int q = blockIdx.y * 8 * J; q < C.n; q += gridDim.y * 8 * J) {
            const int n = C.n - q;
            if (n > 4 * J) tile_rows<TF, TX, 1, 4, J>(tile_smem, a, it, C, q, fac, in, out);
            else if (n > 2 * J) tile_rows<TF, TX, 1, 2, J>(tile_smem, a, it, C, q, fac, in, out);
            else if (n > 2 * H) tile_rows<TF, TX, 1, 1, J>(tile_smem, a, it, C, q, fac, in, out);
            else tile_rows<TF, TX, 1, 1, H>(tile_smem, a, it, C, q, fac, in, out);
        }
    } else {
        const int cw = kWide<TF> ? 4 : it.rows > 2 * kTM2<TF> ? 1 : it.rows > kTM2<TF> ? 2 : 4, tn = 2 * J * cw;
        for (int q = blockIdx.y * tn; q < C.n; q += gridDim.y * tn) {
            const bool half = C.n - q <= 2 * H * cw;
            if constexpr (kWide<TF>) {
                if (half) tile_rows<TF, TX, 2, 1, H>(tile_smem, a, it, C, q, fac, in, out);
                else tile_rows<TF, TX, 2, 1, J>(tile_smem, a, it, C, q, fac, in, out);
            } else if (cw == 1) {
                if (half) tile_rows<TF, TX, 2, 4, H>(tile_smem, a, it, C, q, fac, in, out);
                else tile_rows<TF, TX, 2, 4, J>(tile_smem, a, it, C, q, fac, in, out);
            } else if (cw == 2) {
                if (half) tile_rows<TF, TX, 2, 2, H>(tile_smem, a, it, C, q, fac, in, out);
                else tile_rows<TF, TX, 2, 2, J>(tile_smem, a, it, C, q, fac, in, out);
            } else {
                if (half) tile_rows<TF, TX, 2, 1, H>(tile_smem, a, it, C, q, fac, in, out);
                else tile_rows<TF, TX, 2, 1, J>(tile_smem, a, it, C, q, fac, in, out);
            }
        }
    }
}

// t of the listed blocks: their segments' parts added in order into the first;
// blockIdx.y = right-hand side of the pass
template <class TX>
__global__ void __launch_bounds__(64) k_tile_seg(const FarBlockDev* __restrict__ blocks, const int* __restrict__ list,
                                                 const long long* __restrict__ toff, int seg, TX* __restrict__ t,
                                                 int64_t ldt) {
    const FarBlockDev B = blocks[list[blockIdx.x]];
    const int nseg = (B.n + seg - 1) / seg;
    TX* tb = t + toff[list[blockIdx.x]] + (int64_t)blockIdx.y * ldt;
    for (int k = threadIdx.x; k < B.rank; k += 64) {
        auto acc = as_acc(tb[k]);
        int g = 1;
        for (; g + 4 <= nseg; g += 4) {
            TX v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = tb[k + (int64_t)(g + u) * B.rank];
#pragma unroll
            for (int u = 0; u < 4; ++u) acc_add(acc, as_acc(v[u]));
        }
        for (; g < nseg; ++g) acc_add(acc, as_acc(tb[k + (int64_t)g * B.rank]));
        store(tb + k, acc);
    }
}

// F[a rows] = sum of the partial products of atom a's (block, slot) entries in
// list order, eight of them in flight; blockIdx.y = right-hand side of the pass
template <class TX, class TO>
__global__ void __launch_bounds__(128) k_tile_sum(const int4* __restrict__ items, const int* __restrict__ csr,
                                                  const long long* __restrict__ pbase, const TX* __restrict__ P,
                                                  int64_t ldp, int np, TO* __restrict__ F, int64_t ldf, int rhs0,
                                                  const int2* __restrict__ colr) {
    using TA = typename AccOf<TX>::t;
    const int c = rhs0 + blockIdx.y;
    const int4 item = items[blockIdx.x];
    const int a = item.x, row = item.y + (int)threadIdx.x;
    if (colr) {
        const int2 cr = colr[item.w];
        if (c < cr.x || c >= cr.y) return;
    }
    if (row >= item.z) return;
    const TX* Pc = P + (int64_t)blockIdx.y * ldp + row;
    TA acc = acc_zero<TA>();
    int e = csr[a];
    const int e1 = csr[a + 1];
    for (; e + 8 <= e1; e += 8) {
        TX v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = Pc[__ldg(pbase + e + u)];
#pragma unroll
        for (int u = 0; u < 8; ++u) acc_add(acc, as_acc(v[u]));
    }
    for (; e < e1; ++e) acc_add(acc, as_acc(Pc[__ldg(pbase + e)]));
    store(F + (int64_t)a * np + row + (int64_t)c * ldf, acc);
}

}  // namespace

// right-hand sides per pass: their partial products stay within kTilePass bytes, or
// sixteen columns' (few columns leave tiles empty: 11 columns of the 27 x 27 graded
// array of 4^3 cubes in double-float, one at a time, took 59 ms).  At most 1024,
// which Cols::member needs.
int tile_pass_cols(int64_t part_total, int nrhs, size_t elem) {
    const size_t per = (size_t)std::max<int64_t>(part_total, 1) * elem;
    return (int)std::min<size_t>(std::min(nrhs, 1024), std::max<size_t>(16, Op::kTilePass / per));
}

// The tile kernels read a factor once per group of columns; the per-block kernels
// once per right-hand side or four of them, but without partial products.  Without
// shared factors (gold atoms on a spiral, 3^3 cubes, us): 2 columns pay, 400 atoms 1192 -> 922;
// one column does not, 500 atoms 795 -> 1206, unless the per-block kernel, a CTA for 128 rows
// of an atom, has too few CTAs to hide its loads: 60 atoms 218 -> 108, 150 339 -> 281,
// 200 395 -> 392, 300 523 -> 651.  (complex128 padding costs more: 3 columns.)  Nor do
// the four launches pay for up to four atoms x four columns, or five atoms x one, where the
// per-block kernels' two have a chain of a few blocks (2 atoms 20.0 -> 10.1 us, 5 20.8 -> 18.1).
bool tile_pays(const Op& op, int nrhs) {
    if (op.fprec != VIE_C128 && (op.N <= 4 ? nrhs <= 4 : op.N == 5 && nrhs == 1)) return false;
    const double least = op.fprec == VIE_C128 || nrhs == 1 ? 3.0 : 2.0;
    const bool few = op.fprec != VIE_C128 && 2 * op.n_p2_items < 3 * op.ctx->n_sm;
    return op.share_mean * nrhs >= least || few;
}

Op::~Op() {
    if (!ctx) return;
    auto& v = ctx->ops;
    v.erase(std::remove(v.begin(), v.end(), this), v.end());
}

bool tile_reserve(Op& op, int nrhs, size_t elem, cudaStream_t s) {
    const size_t rp = tile_pass_cols(op.part_total, nrhs, elem);
    const size_t np = (size_t)std::max<int64_t>(op.part_total, 1) * rp * elem;
    const size_t nt = (size_t)std::max<int64_t>(op.ct_total, 1) * rp * elem;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    VIE_CUDA(cudaStreamIsCapturing(s, &cap));
    const bool capturing = cap != cudaStreamCaptureStatusNone;
    if (op.d_part.bytes >= np && op.d_ct.bytes >= nt) {
        op.tile_pinned |= capturing;
        return true;
    }
    if (capturing || (op.tile_oom && np + nt >= op.tile_oom)) return false;
    try {
        if (np + nt > ((size_t)256 << 20) && !op.ctx->admitted) {  // leave 1 GiB to the solver, as ws_pack does
            size_t free_b = 0, total_b = 0;
            VIE_CUDA(cudaMemGetInfo(&free_b, &total_b));
            if (np + nt + ((size_t)1 << 30) > free_b + op.d_part.bytes + op.d_ct.bytes)
                fail(VIE_ERR_OOM, "no room for the register tiles' scratch");
        }
        if (op.d_part.bytes < np) op.d_part.alloc(np);
        if (op.d_ct.bytes < nt) op.d_ct.alloc(nt);
    } catch (const Error& e) {
        if (e.status != VIE_ERR_OOM) throw;
        if (!op.tile_pinned) {
            op.d_part.release();
            op.d_ct.release();
        }
        if (op.ctx->admitted) throw;
        op.tile_oom = np + nt;
        return false;
    }
    return true;
}

bool give_back_scratch(Ctx& c) {
    cudaStreamSynchronize(c.stream);  // (what the failed call had started)
    bool any = false;
    for (Op* o : c.ops) {
        for (DevBuf* b : {&o->d_pw, &o->d_fpart, &o->d_fI, &o->d_fdirs, &o->d_fout}) {
            any |= b->bytes > 0;
            b->release();
        }
        const size_t held = o->d_part.bytes + o->d_ct.bytes;
        if (o->tile_pinned || held == 0) continue;
        o->d_part.release();
        o->d_ct.release();
        o->tile_oom = o->tile_oom ? std::min(o->tile_oom, held) : held;
        any = true;
    }
    return any;
}

template <class TF, class TX, class TO>
void apply_far_tile(Op& op, const TX* x, int64_t ldx, TO* F, int64_t ldf, int nrhs, cudaStream_t s, int first,
                    int count) {
    const int last = count < 0 ? nrhs : first + count;
    const int rp = tile_pass_cols(op.part_total, last - first, sizeof(TX));
    TX* t = op.d_ct.as<TX>();
    TX* P = op.d_part.as<TX>();
    constexpr size_t smem1 = smem_bytes<TF, TX>(1), smem2 = smem_bytes<TF, TX>(2);
    static std::atomic<unsigned long long> attr_set{0};  // devices whose kernels have their shared-memory size
    const unsigned long long bit = 1ull << (op.ctx->device & 63);
    if (!(attr_set.load() & bit)) {
        VIE_CUDA(cudaFuncSetAttribute(k_tile<TF, TX, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem1));
        VIE_CUDA(cudaFuncSetAttribute(k_tile<TF, TX, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem2));
        attr_set.fetch_or(bit);
    }
    for (int c0 = first; c0 < last; c0 += rp) {
        const int nc = std::min(rp, last - c0);
        const bool longest = op.tile_long && (kWide<TF> || (kE<TX> > 1 && nc <= 2));  // (build_apply_lists)
        TileArgs a{op.d_block_atoms.as<int>(), (longest ? op.d_c1_long : op.d_c1_items).as<FarTile>(),
                   op.d_cmem.as<FarMember>(), op.colr, op.np, c0, nc, ldx, op.ct_total, op.part_total};
        const unsigned gy = (unsigned)std::min((op.tile_group * nc + 8 * kJ<TX> - 1) / (8 * kJ<TX>), 65535);
        if (op.n_c1_items > 0) {
            k_tile<TF, TX, 1><<<dim3(op.n_c1_items, gy), kThr, smem1, s>>>(a, op.fac<TF>(), x, t);
            VIE_CHECK_LAUNCH();
        }
        if (op.n_cseg > 0) {
            k_tile_seg<TX><<<dim3(op.n_cseg, nc), 64, 0, s>>>(op.d_blocks.as<FarBlockDev>(), op.d_cseg.as<int>(),
                                                             op.d_ctoff.as<long long>(), op.tile_seg, t, op.ct_total);
            VIE_CHECK_LAUNCH();
        }
        if (op.n_c2_items > 0) {
            a.items = (longest ? op.d_c2_long : op.d_c2_items).as<FarTile>();
            k_tile<TF, TX, 2><<<dim3(op.n_c2_items, gy), kThr, smem2, s>>>(a, op.fac<TF>(), t, P);
            VIE_CHECK_LAUNCH();
        }
        k_tile_sum<TX, TO><<<dim3(op.n_p2_items, nc), 128, 0, s>>>(
            op.d_p2_items.as<int4>(), op.d_p2_csr.as<int>(), op.d_pbase.as<long long>(), P, op.part_total, op.np, F, ldf,
            c0, op.colr);
        VIE_CHECK_LAUNCH();
    }
}

template void apply_far_tile<float2, float2, float2>(Op&, const float2*, int64_t, float2*, int64_t, int, cudaStream_t,
                                                     int, int);
template void apply_far_tile<float2, float4, double2>(Op&, const float4*, int64_t, double2*, int64_t, int, cudaStream_t,
                                                      int, int);
template void apply_far_tile<double2, double2, double2>(Op&, const double2*, int64_t, double2*, int64_t, int,
                                                        cudaStream_t, int, int);

}  // namespace vie
