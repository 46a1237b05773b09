// Far-apply variants and the autotuner that chooses between them.
//
// The far part of a complex float32 apply has several implementations: the
// SIMT kernels with 1, 2, 4 or 8 right-hand sides per factor read, the
// register-tile kernels over the columns (translated copies x right-hand sides)
// of a factor, and for split-precision requests the
// warp-MMA and the tcgen05 tensor-core kernels.  Which is fastest depends on the right-hand-side count
// and on the operator (rank distribution, atom size), so the choice is made by
// timing on the operator itself and is remembered per power-of-two bucket of
// the right-hand-side count.
#include <algorithm>
#include <cmath>

#include "common.h"

namespace vie {

namespace {

int bucket(int nrhs) {
    int b = 0;
    while ((2 << b) <= nrhs && b < 30) ++b;
    return b;
}

bool admissible(int precision, int v) {
    if ((v >= VIE_VAR_SIMT_R1 && v <= VIE_VAR_SIMT_R8) || v == VIE_VAR_SIMT_SHARED) return true;
    return precision == VIE_BF16X3 &&
           (v == VIE_VAR_MMA_BF16X3 || v == VIE_VAR_TCGEN05_BF16X3 || v == VIE_VAR_TCGEN05_PACKED_BF16X3 ||
            v == VIE_VAR_TCGEN05_WS_BF16X3 || v == VIE_VAR_TCGEN05_WS2_BF16X3);
}

int default_variant(Op& op, int precision, int nrhs) {
    // BF16x3: the warp-specialised kernel, with two row tiles per B tile above 32
    // columns, where gathering and splitting B weighs most, else as its lists balance
    if (precision == VIE_BF16X3 && nrhs >= 8) {
        if (nrhs <= 32) build_ws_lists(op);
        return nrhs <= 32 && op.ws_tiles == 1 ? VIE_VAR_TCGEN05_WS_BF16X3 : VIE_VAR_TCGEN05_WS2_BF16X3;
    }
    return nrhs == 1 ? (tile_pays(op, 1) ? VIE_VAR_SIMT_SHARED : VIE_VAR_SIMT_R1) : VIE_VAR_SIMT_R4;
}

// the variants that read a factor once per group of right-hand sides: the
// register tiles take all columns (copies x right-hand sides) of a factor
// together where that pays, in one summation order for the three group sizes
void far_grouped(Op& op, const float2* x, int64_t ldx, float2* F, int64_t ldf, int nrhs, int nr, int precision,
                 cudaStream_t s) {
    if (far_tiled(op, precision, nrhs) && tile_reserve(op, nrhs, sizeof(float2), s))
        apply_far_tile<float2, float2, float2>(op, x, ldx, F, ldf, nrhs, s);
    else
        apply_far_simt32(op, x, ldx, F, ldf, nrhs, nr, s);
}

}  // namespace

int far_variant(Op& op, int precision, int nrhs) {
    auto it = op.variant.find({precision, bucket(nrhs)});
    return it != op.variant.end() ? it->second : default_variant(op, precision, nrhs);
}

bool far_tiled(const Op& op, int precision, int nrhs) {
    const auto it = op.tiled.find({precision, bucket(nrhs)});
    return it != op.tiled.end() ? it->second : tile_pays(op, nrhs);
}

void far32(Op& op, const float2* x, int64_t ldx, float2* F, int64_t ldf, int nrhs, int precision, cudaStream_t s) {
    switch (far_variant(op, precision, nrhs)) {
        case VIE_VAR_SIMT_R1: apply_far_simt32(op, x, ldx, F, ldf, nrhs, 1, s); break;
        case VIE_VAR_SIMT_R2: far_grouped(op, x, ldx, F, ldf, nrhs, 2, precision, s); break;
        case VIE_VAR_SIMT_R4: far_grouped(op, x, ldx, F, ldf, nrhs, 4, precision, s); break;
        case VIE_VAR_SIMT_R8: far_grouped(op, x, ldx, F, ldf, nrhs, 8, precision, s); break;
        case VIE_VAR_MMA_BF16X3: apply_far_bf16x3(op, x, ldx, F, ldf, nrhs, s); break;
        case VIE_VAR_TCGEN05_BF16X3: apply_far_umma(op, x, ldx, F, ldf, nrhs, s); break;
        case VIE_VAR_TCGEN05_PACKED_BF16X3: apply_far_umma_packed(op, x, ldx, F, ldf, nrhs, s); break;
        case VIE_VAR_SIMT_SHARED:
            // one right-hand side at a time: a column's result does not depend on the others
            for (int c = 0; c < nrhs; ++c) {
                if (tile_reserve(op, 1, sizeof(float2), s))
                    apply_far_tile<float2, float2, float2>(op, x, ldx, F, ldf, nrhs, s, c, 1);
                else
                    apply_far_simt32(op, x + c * ldx, ldx, F + c * ldf, ldf, 1, 1, s);
            }
            break;
        case VIE_VAR_TCGEN05_WS_BF16X3: apply_far_umma_ws(op, x, ldx, F, ldf, nrhs, s); break;
        case VIE_VAR_TCGEN05_WS2_BF16X3: apply_far_umma_ws2(op, x, ldx, F, ldf, nrhs, s); break;
        default: fail(VIE_ERR_STATE, "unknown far-apply variant");
    }
}

int tune_far(Op& op, int precision, int nrhs, cudaStream_t s, std::vector<int>& cand, std::vector<double>& ms) {
    if (op.fprec != VIE_C64) fail(VIE_ERR_INVALID_ARG, "vie_tune: needs VIE_C64 factors");
    if (precision != VIE_C64 && precision != VIE_BF16X3) fail(VIE_ERR_INVALID_ARG, "vie_tune: VIE_C64 or VIE_BF16X3");
    if (nrhs < 1 || nrhs > 1024) fail(VIE_ERR_INVALID_ARG, "vie_tune: 1 to 1024 right-hand sides");
    cand.clear();
    ms.clear();
    for (int v = VIE_VAR_SIMT_R1; v <= VIE_VAR_TCGEN05_WS2_BF16X3; ++v) {
        if (!admissible(precision, v)) continue;
        if (v >= VIE_VAR_SIMT_R2 && v <= VIE_VAR_SIMT_R8 && nrhs == 1) continue;  // same as R1
        if (v == VIE_VAR_SIMT_SHARED && nrhs > 1) continue;  // one column at a time
        cand.push_back(v);
    }
    const int64_t n = op.n();
    DevBuf x((size_t)n * nrhs * sizeof(float2)), F((size_t)n * nrhs * sizeof(float2));
    VIE_CUDA(cudaMemsetAsync(x.p, 0, (size_t)n * nrhs * sizeof(float2), s));
    // the planes of 9 and 10 first: those of 7, one set per block, are many times larger, and
    // stay only if 7 is chosen (or was before)
    struct PackGuard {
        Op& o;
        bool keep;
        ~PackGuard() {
            if (keep) return;
            o.d_u1_pack.release();
            o.d_u2_pack.release();
            o.umma_packed = false;
        }
    } packed{op, op.umma_packed || precision != VIE_BF16X3};
    if (precision == VIE_BF16X3) {
        ws_pack(op, s);
        umma_prepare(op, s);
        try {
            umma_pack(op, s);
        } catch (const Error& e) {  // no room beside the others: 7 is timed as 6
            if (!e.memory) throw;
            op.umma_pack_failed = true;
        }
    }
    cudaEvent_t e0, e1;
    VIE_CUDA(cudaEventCreate(&e0));
    VIE_CUDA(cudaEventCreate(&e1));
    // time all columns of the operator (a batched solve's column table does not apply here)
    struct ColrGuard {
        Op& o;
        const int2* saved;
        ~ColrGuard() { o.colr = saved; }
    } guard{op, op.colr};
    op.colr = nullptr;
    const auto key = std::make_pair(precision, bucket(nrhs));
    const auto had_variant = op.variant.find(key) != op.variant.end() ? op.variant[key] : 0;
    const auto had_form = op.tiled;
    int best = 0;
    bool best_form = false;
    double best_ms = 1e300;
    auto time_one = [&] {
        far32(op, x.as<float2>(), n, F.as<float2>(), n, nrhs, precision, s);  // warm-up
        double t = 1e300;
        for (int r = 0; r < 3; ++r) {
            VIE_CUDA(cudaEventRecord(e0, s));
            far32(op, x.as<float2>(), n, F.as<float2>(), n, nrhs, precision, s);
            VIE_CUDA(cudaEventRecord(e1, s));
            VIE_CUDA(cudaEventSynchronize(e1));
            float m = 0.f;
            VIE_CUDA(cudaEventElapsedTime(&m, e0, e1));
            t = std::min(t, (double)m);
        }
        return t;
    };
    try {
        for (int v : cand) {
            op.variant[key] = v;
            // R2, R4, R8 as per-block kernels; the register tiles, one kernel for the
            // three, beside R4
            const bool grouped = v >= VIE_VAR_SIMT_R2 && v <= VIE_VAR_SIMT_R8;
            double t = 1e300;
            for (int form = 0; form < (v == VIE_VAR_SIMT_R4 ? 2 : 1); ++form) {
                if (grouped) op.tiled[key] = form == 1;
                const double tf = time_one();
                t = std::min(t, tf);
                if (tf < best_ms) {
                    best_ms = tf;
                    best = v;
                    best_form = form == 1;
                }
            }
            ms.push_back(t);
        }
    } catch (...) {
        if (had_variant) op.variant[key] = had_variant;
        else op.variant.erase(key);
        op.tiled = had_form;
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
        throw;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    packed.keep |= best == VIE_VAR_TCGEN05_PACKED_BF16X3;
    op.variant[key] = best;
    if (best >= VIE_VAR_SIMT_R2 && best <= VIE_VAR_SIMT_R8) op.tiled[key] = best_form;
    else op.tiled.erase(key);
    return best;
}

int tune_entry(Op& op, int precision, int nrhs, int force, vie_tune_result* res, cudaStream_t s) {
    std::vector<int> cand;
    std::vector<double> ms;
    int v;
    if (force > 0) {
        if (!admissible(precision, force)) fail(VIE_ERR_INVALID_ARG, "vie_tune: variant not admissible for precision");
        if (op.fprec != VIE_C64) fail(VIE_ERR_INVALID_ARG, "vie_tune: needs VIE_C64 factors");
        if (nrhs < 1 || nrhs > 1024) fail(VIE_ERR_INVALID_ARG, "vie_tune: 1 to 1024 right-hand sides");
        op.variant[{precision, bucket(nrhs)}] = force;
        op.tiled.erase({precision, bucket(nrhs)});
        v = force;
    } else {
        v = tune_far(op, precision, nrhs, s, cand, ms);
    }
    if (res) {
        res->variant = v;
        res->n_candidates = (int)std::min<size_t>(16, cand.size());
        for (int i = 0; i < res->n_candidates; ++i) {
            res->candidates[i] = cand[i];
            res->ms[i] = ms[i];
        }
    }
    return VIE_OK;
}

bool tuned(const Op& op, int precision, int nrhs) { return op.variant.count({precision, bucket(nrhs)}) > 0; }

}  // namespace vie
