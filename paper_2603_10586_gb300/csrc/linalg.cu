#include <algorithm>
// Dense kernels around the self blocks (paper Sec. 4, eq. diagprecond):
// explicit inverse of each distinct Z_ii by Gauss-Jordan elimination with
// partial pivoting (float64), precision conversions, and the per-type block
// product Y = M B (+ A) over all atoms of one type (the self part of the
// operator, the preconditioner and the fused P^-1 Z form).
#include "common.h"
#include "cplx.cuh"
#include "tilemma.cuh"

namespace vie {

namespace {

// ---------------------------------------------------------------------------
// Inverse of one np x np self block: in-place Gauss-Jordan elimination with
// partial pivoting, one cooperative launch.  CTA b holds the columns b, b + G,
// ... (in shared memory when they fit, else in `work`) for the whole
// elimination, so a step moves only the next pivot column: its owner writes the
// updated column to cb[(k + 1) & 1] while the others still read cb[k & 1], and one
// grid barrier per step separates them.  Every CTA finds the pivot of the column
// by itself.  A step is np^2 / G complex products per CTA, well under a
// microsecond, so the barrier and the pivot search bound it.  (Two kernels per
// step through memory, on the augmented matrix, took 1.67 ms at np = 108; this
// takes 0.55 ms.)
// The row swaps of the pivoting leave the inverse's columns permuted; `perm`
// undoes that at the end.  The barrier's waits are bounded (status 2): a grid that gave
// up is run again as one CTA, which waits for nobody, so a GPU that is kept busy for
// longer by other work costs time and not the call.
// ---------------------------------------------------------------------------
constexpr int kGjThr = 256;
constexpr size_t kGjSmemMax = 200 * 1024;
constexpr long long kGjWaitCycles = 2000000000LL;  // ~1 s

__device__ __forceinline__ bool gj_barrier(unsigned* ctr, unsigned target, int* status, long long lim) {
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(ctr, 1u);
        const long long t0 = clock64();
        ok = 1;
        unsigned v;
        do {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ctr) : "memory");
            if (v < target && clock64() - t0 >= lim) {
                atomicExch(status, 2);
                ok = 0;
                break;
            }
        } while (v < target);
    }
    __syncthreads();
    return ok != 0;
}

__global__ void __launch_bounds__(kGjThr) k_gj_inverse(const double2* __restrict__ A, double2* __restrict__ inv, int np,
                                                       int max_cols, double2* cb, double2* work, int* piv, int* perm,
                                                       unsigned* ctr, int* status, long long lim) {
    extern __shared__ __align__(16) unsigned char gj_smem[];
    const int G = gridDim.x, b = blockIdx.x, tid = threadIdx.x;
    const int nc = (np - b + G - 1) / G;  // columns of this CTA: b + c G
    double2* scol = reinterpret_cast<double2*>(gj_smem);
    double2* srow = scol + (work ? 0 : np);                      // r, then the old row k, per column
    double2* M = work ? work + (size_t)b * max_cols * np : srow + 2 * max_cols;
    __shared__ double best[kGjThr / 32];
    __shared__ int bidx[kGjThr / 32];
    for (int e = tid; e < nc * np; e += kGjThr) {
        const int c = e / np, i = e - c * np;
        const double2 v = A[i + (size_t)(b + c * G) * np];
        M[e] = v;
        if (b + c * G == 0) cb[i] = v;
    }
    unsigned target = G;
    if (!gj_barrier(ctr, target, status, lim)) return;
    for (int k = 0; k < np; ++k) {
        const double2* col = cb + (size_t)(k & 1) * np;
        double bv = -1.0;
        int bi = k;
        for (int i = tid; i < np; i += kGjThr) {
            const double2 v = __ldcg(col + i);
            if (!work) scol[i] = v;
            const double a = v.x * v.x + v.y * v.y;
            if (i >= k && a > bv) { bv = a; bi = i; }
        }
        for (int o = 16; o > 0; o >>= 1) {
            const double ov = __shfl_down_sync(0xffffffffu, bv, o);
            const int oi = __shfl_down_sync(0xffffffffu, bi, o);
            if (ov > bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
        }
        if ((tid & 31) == 0) { best[tid >> 5] = bv; bidx[tid >> 5] = bi; }
        __syncthreads();
        bv = best[0];
        bi = bidx[0];
        for (int w = 1; w < kGjThr / 32; ++w)
            if (best[w] > bv || (best[w] == bv && bidx[w] < bi)) { bv = best[w]; bi = bidx[w]; }
        const int p = bi;
        if (!(bv > 0.0)) {  // singular: the same decision in every CTA
            if (tid == 0) *status = 1;
            return;
        }
        if (b == 0 && tid == 0) piv[k] = p;
        auto colv = [&](int i) { return work ? __ldcg(col + i) : scol[i]; };
        const double2 pv = colv(p), ck = colv(k);
        const double den = 1.0 / (pv.x * pv.x + pv.y * pv.y);
        const double2 ip = make_double2(pv.x * den, -pv.y * den);
        for (int c = tid; c < nc; c += kGjThr) {
            srow[c] = b + c * G == k ? ip : cmul(M[(size_t)c * np + p], ip);
            srow[max_cols + c] = M[(size_t)c * np + k];
        }
        __syncthreads();
        double2* next = cb + (size_t)((k + 1) & 1) * np;
        for (int e = tid; e < nc * np; e += kGjThr) {
            const int c = e / np, i = e - c * np, j = b + c * G;
            const double2 r = srow[c];
            double2 v;
            if (i == k) {
                v = r;
            } else {
                // rows k and p swapped: row p holds the old row k
                const double2 f = i == p ? ck : colv(i);
                v = j == k ? make_double2(0.0, 0.0) : i == p ? srow[max_cols + c] : M[e];
                v.x -= f.x * r.x - f.y * r.y;
                v.y -= f.x * r.y + f.y * r.x;
            }
            M[e] = v;
            if (j == k + 1) next[i] = v;
        }
        target += G;
        if (!gj_barrier(ctr, target, status, lim)) return;
    }
    // column k of the inverse: undo the swaps, last first
    if (b == 0 && tid == 0) {
        for (int j = 0; j < np; ++j) perm[j] = j;
        for (int k = np - 1; k >= 0; --k) {
            const int p = piv[k], t = perm[k];
            perm[k] = perm[p];
            perm[p] = t;
        }
        for (int j = 0; j < np; ++j) perm[np + perm[j]] = j;
    }
    target += G;
    if (!gj_barrier(ctr, target, status, lim)) return;
    for (int e = tid; e < nc * np; e += kGjThr) {
        const int c = e / np, i = e - c * np;
        inv[i + (size_t)__ldcg(perm + np + b + c * G) * np] = M[e];
    }
}

__global__ void c128_to_c64(const double2* s, float2* d, int64_t n) {
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n) d[t] = make_float2((float)s[t].x, (float)s[t].y);
}
__global__ void c64_to_c128(const float2* s, double2* d, int64_t n) {
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n) d[t] = make_double2(s[t].x, s[t].y);
}

// ---------------------------------------------------------------------------
// Y[:, col] = M B[:, col] (+ ADD[:, col]) for the columns col = (atom of the
// type, rhs).  M: np x np column-major.  Vector element (row r of atom a, rhs c)
// lives at a * np + r + c * ld.  A CTA of four warps takes 16 RA rows x 2 J WN
// columns, the warps side by side and, where the columns are few, along K (WK =
// 4 / WN groups added in order at the end); operands staged by cp.async through two
// shared-memory buffers.  Bound by the float32 (float64) pipes; self_gemm
// picks the width.  (A 2 x 2 sub-tile per
// thread and 32 x 32 per CTA, the kernel before, took 997 us for 61,440 columns of
// np = 240 in float32, now 669 us, and 19 us for 16 columns of np = 108, now 9 us.)
// ADD may be Y itself (y = Z_ii x + y in place): every output element is read
// from ADD and then written to Y by the one thread that owns it, so ADD and Y
// carry no __restrict__ and ADD is read through the ordinary (coherent) path.
// B must not overlap Y.
// ---------------------------------------------------------------------------
constexpr int kGemmThr = 128;
template <class T, int WN, int RA, int J, int K = RA == 2 ? 512 / (int)sizeof(T) : 16>
struct GemmShape {
    static constexpr int WK = 4 / WN, TM = 16 * RA, TN = 2 * J * WN;
    // (K: the narrow tile of small arrays takes its K range in few, longer stages: their
    // latency is all there is)
    static constexpr int KC = K, KG = KC / WK;
    static constexpr int LA = TM, LB = KC + kE<T>;  // A [K][row], B [column][K]
    static constexpr size_t a_pad = (size_t)KC * LA * sizeof(T);
    static constexpr size_t stage = a_pad + (size_t)TN * LB * sizeof(T);
};

template <class T, int WN, int RA, int J, int K>
__global__ void __launch_bounds__(kGemmThr, 3) type_gemm(const T* __restrict__ M, int np, int tile_rows,
                                                         const int* __restrict__ atoms, int n_atoms, int nrhs,
                                                         const T* __restrict__ B, int64_t ldb, const T* ADD,
                                                         int64_t ldadd, T* Y, int64_t ldy,
                                                         const int2* __restrict__ colr, int prob) {
    using S = GemmShape<T, WN, RA, J, K>;
    constexpr int E = kE<T>, UR = S::TM / E, UK = S::KC / E;   // 16-byte units per K value of A, per column of B
    constexpr int KA = kGemmThr / UR, CB = kGemmThr / UK;      // K values of A, columns of B staged at a time
    constexpr int NB = (S::TN + CB - 1) / CB;
    __shared__ __align__(16) unsigned char smem[2 * S::stage];
    // right-hand sides of this type's problem (all of them for a single operator)
    const int2 cr = colr ? colr[prob] : make_int2(0, nrhs);
    const int ncols = n_atoms * (cr.y - cr.x);
    const int row0 = blockIdx.x * tile_rows, rows = min(tile_rows, np - row0), col0 = blockIdx.y * S::TN;
    if (col0 >= ncols) return;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int wn = warp % WN, wk = warp / WN, tr = lane & 15, tc = lane >> 4;
    const int ur = tid % UR * E, uk = tid / UR, kb = tid % UK * E, cb = tid / UK;
    const T* Ms = M + row0 + ur + (int64_t)uk * np;
    const T* bs[NB];
    unsigned live = 0;
#pragma unroll
    for (int u = 0; u < NB; ++u) {
        const int q = cb + u * CB, gc = col0 + q;
        const bool ok = q < S::TN && gc < ncols;
        bs[u] = ok ? B + (int64_t)atoms[gc % n_atoms] * np + kb + (int64_t)(cr.x + gc / n_atoms) * ldb : B;
        live |= ok ? 1u << u : 0u;
    }
    const int nst = (np + S::KC - 1) / S::KC;
    auto fill = [&](int s) {
        T* As = reinterpret_cast<T*>(smem + (s & 1) * S::stage) + uk * S::LA + ur;
        T* Bs = reinterpret_cast<T*>(smem + (s & 1) * S::stage + S::a_pad) + cb * S::LB + kb;
#pragma unroll
        for (int k = 0; k < S::KC; k += KA) {
            const bool ok = s * S::KC + k + uk < np && ur < rows;
            if (KA <= S::KC || uk < S::KC)
                cp_async16(As + k * S::LA, ok ? Ms + (int64_t)(s * S::KC + k) * np : M, ok);
        }
#pragma unroll
        for (int u = 0; u < NB; ++u)
            if (cb + u * CB < S::TN) {
                const bool ok = ((live >> u) & 1) && s * S::KC + kb < np;
                cp_async16(Bs + u * CB * S::LB, ok ? bs[u] + s * S::KC : B, ok);
            }
        cp_commit();
    };
    T acc[RA][J];
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
        mma_stage<T, T, T, 2, S::KG, S::LA, S::LB, RA, J>(
            reinterpret_cast<const T*>(st) + wk * S::KG * S::LA + E * tr,
            reinterpret_cast<const T*>(st + S::a_pad) + (wn * 2 * J + tc) * S::LB + wk * S::KG, acc);
        __syncthreads();
    }
    if (S::WK > 1) {
        T* buf = reinterpret_cast<T*>(smem);
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
                    for (int j = 0; j < J; ++j) acc[i][j] += buf[((wn * RA + i) * J + j) * 32 + lane];
            __syncthreads();
        }
    }
    if (wk == 0)
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const int gc = col0 + wn * 2 * J + tc + 2 * j;
            if (gc >= ncols) continue;
            const int64_t at = (int64_t)atoms[gc % n_atoms] * np + row0, rhs = cr.x + gc / n_atoms;
#pragma unroll
            for (int i = 0; i < RA; ++i) {
                const int r = E == 2 ? 32 * (i >> 1) + 2 * tr + (i & 1) : 16 * i + tr;
                if (r >= rows) continue;
                T v = acc[i][j];
                if (ADD) v += ADD[at + r + rhs * ldadd];
                Y[at + r + rhs * ldy] = v;
            }
        }
}

}  // namespace

// all types' inverses with G CTAs each; returns the kernels' status
static int gj_run(Op& op, int G, cudaStream_t s) {
    const int np = op.np, max_cols = (np + G - 1) / G;
    size_t smem = ((size_t)np + 2 * max_cols + (size_t)max_cols * np) * sizeof(double2);
    const bool in_smem = smem <= kGjSmemMax;
    if (!in_smem) smem = 2 * (size_t)max_cols * sizeof(double2);
    VIE_CUDA(cudaFuncSetAttribute(k_gj_inverse, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGjSmemMax));
    // one allocation: the two pivot columns, the CTAs' columns when they are not in
    // shared memory, then pivots, permutation, status and one barrier counter per type
    const size_t nz = 2 * (size_t)np + (in_smem ? 0 : (size_t)G * max_cols * np);
    const size_t ni = 3 * (size_t)np + 1 + op.T;
    TmpBuf buf(nz * sizeof(double2) + ni * sizeof(int));
    double2* cb = buf.as<double2>();
    double2* work = in_smem ? nullptr : cb + 2 * (size_t)np;
    int* piv = reinterpret_cast<int*>(cb + nz);
    int* perm = piv + np;
    int* status = perm + 2 * (size_t)np;
    unsigned* ctr = reinterpret_cast<unsigned*>(status + 1);
    long long lim = wait_limit(kGjWaitCycles);
    VIE_CUDA(cudaMemsetAsync(status, 0, (1 + op.T) * sizeof(int), s));
    for (int t = 0; t < op.T; ++t) {
        const double2* A = op.d_zself64.as<double2>() + (size_t)t * np * np;
        double2* Inv = op.d_inv64.as<double2>() + (size_t)t * np * np;
        unsigned* c = ctr + t;
        int n = np, mc = max_cols;
        void* args[] = {&A, &Inv, &n, &mc, &cb, &work, &piv, &perm, &c, &status, &lim};
        VIE_CUDA(cudaLaunchCooperativeKernel((const void*)k_gj_inverse, dim3(G), dim3(kGjThr), args, smem, s));
        VIE_CHECK_LAUNCH();
    }
    int st = 0;
    VIE_CUDA(cudaMemcpyAsync(&st, status, sizeof(int), cudaMemcpyDeviceToHost, s));
    VIE_CUDA(cudaStreamSynchronize(s));
    return st;
}

void invert_self_blocks(Op& op) {
    cudaStream_t s = op.ctx->stream;
    op.d_inv64.alloc((size_t)op.T * op.np * op.np * sizeof(double2));
    // two columns per CTA, or as many as one CTA per SM leaves
    int st = gj_run(op, std::min(op.ctx->n_sm, (op.np + 1) / 2), s);
    if (st == 2) st = gj_run(op, 1, s);
    if (st) fail(VIE_ERR_BREAKDOWN, "a meta-atom self block is singular");
}

void convert_c128_to_c64(const void* src, void* dst, int64_t n, cudaStream_t s) {
    if (n <= 0) return;
    c128_to_c64<<<(unsigned)((n + 255) / 256), 256, 0, s>>>((const double2*)src, (float2*)dst, n);
    VIE_CHECK_LAUNCH();
}
void convert_c64_to_c128(const void* src, void* dst, int64_t n, cudaStream_t s) {
    if (n <= 0) return;
    c64_to_c128<<<(unsigned)((n + 255) / 256), 256, 0, s>>>((const float2*)src, (double2*)dst, n);
    VIE_CHECK_LAUNCH();
}

template <class T2>
__global__ void k_conj(const T2* src, T2* dst, int64_t n) {  // may run in place
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const T2 v = src[i];
        dst[i] = mk(v.x, -v.y);
    }
}

template <class T2>
__global__ void k_conj_transpose(const T2* __restrict__ src, T2* __restrict__ dst, int np) {
    const int64_t base = (int64_t)blockIdx.y * np * np;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < (int64_t)np * np;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = e % np, c = e / np;
        const T2 v = src[base + c + r * np];  // element (c, r) of the source
        dst[base + e] = mk(v.x, -v.y);
    }
}

void conj_copy(const void* src, void* dst, int64_t n, bool c128, cudaStream_t s) {
    if (n <= 0) return;
    const unsigned g = (unsigned)std::min<int64_t>(8192, (n + 255) / 256);
    if (c128) k_conj<double2><<<g, 256, 0, s>>>((const double2*)src, (double2*)dst, n);
    else k_conj<float2><<<g, 256, 0, s>>>((const float2*)src, (float2*)dst, n);
    VIE_CHECK_LAUNCH();
}

void conj_transpose_blocks(const void* src, void* dst, int T, int np, bool c128, cudaStream_t s) {
    const dim3 g((unsigned)std::min<int64_t>(1024, ((int64_t)np * np + 255) / 256), T);
    if (c128) k_conj_transpose<double2><<<g, 256, 0, s>>>((const double2*)src, (double2*)dst, np);
    else k_conj_transpose<float2><<<g, 256, 0, s>>>((const float2*)src, (float2*)dst, np);
    VIE_CHECK_LAUNCH();
}

namespace {
template <class T, int WN, int RA, int J, int K = GemmShape<T, WN, RA, J>::KC>
void launch_gemm(const T* M, int np, const int* atoms, int na, int nrhs, const T* B, int64_t ldb, const T* ADD,
                 int64_t ldadd, T* Y, int64_t ldy, const int2* colr, int prob, cudaStream_t s) {
    using S = GemmShape<T, WN, RA, J, K>;
    const int nt = (np + S::TM - 1) / S::TM, tile_rows = ((np + nt - 1) / nt + 1) / 2 * 2;  // equal, even pieces
    const dim3 grid((np + tile_rows - 1) / tile_rows, (unsigned)(((int64_t)na * nrhs + S::TN - 1) / S::TN));
    type_gemm<T, WN, RA, J, K><<<grid, kGemmThr, 0, s>>>(M, np, tile_rows, atoms, na, nrhs, B, ldb, ADD, ldadd, Y, ldy,
                                                      colr, prob);
    VIE_CHECK_LAUNCH();
}
}  // namespace

// mode 0: Y = M X + C   (self part plus far part C)
// mode 1: Y = X + M C   (fused preconditioner: X + Z_D^-1 (far part))
// mode 2: Y = M X       (plain block product, e.g. the preconditioner)
template <class TM, class TX>
void self_gemm(Op& op, const TM* M, const TX* X, int64_t ldx, const TX* C, int64_t ldc, TX* Y, int64_t ldy,
               int nrhs, int mode, cudaStream_t s) {
    const int np = op.np;
    constexpr int J = sizeof(TX) == 8 ? 8 : 4;
    for (int t = 0; t < op.T; ++t) {
        int na = op.type_atom_off[t + 1] - op.type_atom_off[t];
        if (na == 0) continue;
        const int* atoms = op.d_atoms_by_type.as<int>() + op.type_atom_off[t];
        const TM* Mt = M + (size_t)t * np * np;
        const TX* Bop = mode == 1 ? C : X;
        int64_t ldb = mode == 1 ? ldc : ldx;
        const TX* ADD = mode == 0 ? C : (mode == 1 ? X : nullptr);
        int64_t ldadd = mode == 0 ? ldc : ldx;
        const int prob = op.type_prob.empty() ? 0 : op.type_prob[t];
        // The widest tile that gives every SM two CTAs; the narrowest (32 rows, four
        // warps along K) when none does.  complex128 keeps its SM's float64 units busy whatever
        // the width, so there the SM with the most columns decides, and of the widths with
        // two CTAs per SM the one with the fewest such columns is taken (a narrower one from 2%
        // on; us: 81 atoms of 240 unknowns x 33 columns 1443 -> 1091, 256 x 16 1920 -> 1681,
        // 49 of 450 x 64 5539 -> 4850; complex float32 loses nothing by its widest tiles).  Blocks
        // of up to 32 rows (one voxel per edge) would leave most of a 64-row tile empty: 32
        // rows x 32 columns (complex128: 16), 16 K values per stage (6 unknowns, 576 atoms x 33
        // columns: 9.0 -> 6.1 us; complex128 131 -> 70 us).
        const int64_t rt = (np + 63) / 64, cols = (int64_t)na * nrhs, want = 2 * op.ctx->n_sm;
        int width = 3;  // 8 J, 4 J or 2 J columns, or the narrowest
        double least = 0.0;
        for (int w = 0; w < 3; ++w) {
            const int tn = 8 * J >> w;
            const int64_t ctas = rt * ((cols + tn - 1) / tn);
            if (ctas < want) continue;
            const int64_t per_sm = (ctas + op.ctx->n_sm - 1) / op.ctx->n_sm;
            const double most = sizeof(TX) == 16 ? (double)(per_sm * tn) * (1.0 + 0.02 * w) : 1.0;
            if (width == 3 || most < least) {
                width = w;
                least = most;
            }
        }
#define VIE_GEMM(WN, RA) \
    launch_gemm<TX, WN, RA, J>(Mt, np, atoms, na, nrhs, Bop, ldb, ADD, ldadd, Y, ldy, op.colr, prob, s)
        if (np <= 32)
            launch_gemm<TX, J / 2, 2, 4, 16>(Mt, np, atoms, na, nrhs, Bop, ldb, ADD, ldadd, Y, ldy, op.colr, prob, s);
        else if (width == 0) VIE_GEMM(4, 4);
        else if (width == 1) VIE_GEMM(2, 4);
        else if (width == 2) VIE_GEMM(1, 4);
        else launch_gemm<TX, 1, 2, 4>(Mt, np, atoms, na, nrhs, Bop, ldb, ADD, ldadd, Y, ldy, op.colr, prob, s);
#undef VIE_GEMM
    }
}

template void self_gemm<float2, float2>(Op&, const float2*, const float2*, int64_t, const float2*, int64_t,
                                        float2*, int64_t, int, int, cudaStream_t);
template void self_gemm<double2, double2>(Op&, const double2*, const double2*, int64_t, const double2*, int64_t,
                                          double2*, int64_t, int, int, cudaStream_t);

}  // namespace vie
