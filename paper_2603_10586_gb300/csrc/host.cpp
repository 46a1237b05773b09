// Host-side algorithms of libvie: voxel/face mesh of an atom type, grid
// hierarchy and far-block lists, the greedy least-loaded work map and the
// work lists of the compressed apply.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdlib>
#include <limits>
#include <map>
#include <mutex>
#include <numeric>
#include <queue>
#include <unordered_map>

#include "common.h"

namespace vie {

std::atomic<long long> g_kernel_launches{0};

void fail(int status, const std::string& msg) { throw Error{status, msg}; }

double now_s() {
    using namespace std::chrono;
    return duration<double>(steady_clock::now().time_since_epoch()).count();
}

long long wait_limit(long long normal) {
    const char* e = std::getenv("VIE_TEST_WAIT_CYCLES");
    return e && *e ? std::max(0LL, std::atoll(e)) : normal;
}

static thread_local Ctx* t_alloc_ctx = nullptr;

AllocScope::AllocScope(Ctx* c) : prev(t_alloc_ctx) { t_alloc_ctx = c; }
AllocScope::~AllocScope() { t_alloc_ctx = prev; }

static thread_local cudaStream_t t_tmp_stream = nullptr;
static thread_local bool t_tmp_on = false;

TmpScope::TmpScope(cudaStream_t s) : prev(t_tmp_stream), prev_on(t_tmp_on) {
    t_tmp_stream = s;
    t_tmp_on = true;
}
TmpScope::~TmpScope() {
    t_tmp_stream = prev;
    t_tmp_on = prev_on;
}

// The open pools of the process: an allocation that the GPU has no room for takes back
// what any of them keeps, not only its own context's.
static std::mutex g_pools_mu;
static std::vector<Ctx*> g_pools;

void Ctx::pool_open() {
    cudaMemPoolProps pp = {};
    pp.allocType = cudaMemAllocationTypePinned;
    pp.handleTypes = cudaMemHandleTypeNone;
    pp.location.type = cudaMemLocationTypeDevice;
    pp.location.id = device;
    if (cudaMemPoolCreate(&pool, &pp) != cudaSuccess) {
        pool = nullptr;
        cudaGetLastError();
        return;
    }
    uint64_t keep = kPoolKeep;
    cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
    std::lock_guard<std::mutex> lk(g_pools_mu);
    g_pools.push_back(this);
}

void Ctx::pool_close() {
    if (!pool) return;
    {
        std::lock_guard<std::mutex> lk(g_pools_mu);
        g_pools.erase(std::find(g_pools.begin(), g_pools.end(), this));
    }
    cudaStreamSynchronize(stream);
    cudaMemPoolDestroy(pool);
    pool = nullptr;
}

void Ctx::pool_trim() {
    if (!pool) return;
    cudaStreamSynchronize(stream);
    cudaMemPoolTrimTo(pool, 0);
}

int64_t Ctx::pool_kept() const {
    uint64_t reserved = 0, used = 0;
    if (!pool || cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReservedMemCurrent, &reserved) != cudaSuccess ||
        cudaMemPoolGetAttribute(pool, cudaMemPoolAttrUsedMemCurrent, &used) != cudaSuccess)
        return 0;
    return std::max<int64_t>(0, (int64_t)reserved - (int64_t)used - kPoolChunk);
}

void DevBuf::alloc(size_t b) {
    release();
    if (b == 0) b = 1;
    Ctx* c = t_alloc_ctx;
    int64_t kept = 0;  // what the pool keeps counts against a cap
    if (c) {
        const int64_t cap = c->cap.load();
        const int64_t now = c->allocated.fetch_add((int64_t)b) + (int64_t)b;
        if (cap > 0) {
            kept = c->pool_kept();
            if (kept > 0 && now + kept > cap) {
                c->pool_trim();
                kept = c->pool_kept();
            }
        }
        if (cap > 0 && now > cap) {
            c->allocated.fetch_sub((int64_t)b);
            throw Error{VIE_ERR_OOM,
                        "allocation of " + std::to_string(b) + " bytes would exceed the context's cap of " +
                            std::to_string(cap) + " bytes",
                        true};
        }
    }
    // (the null stream names no stream to free on: such a buffer is not pooled)
    const bool pooled = tmp && t_tmp_on && t_tmp_stream && c && c->pool && b <= TmpBuf::kPoolMax;
    cudaError_t e = pooled ? cudaMallocFromPoolAsync(&p, b, c->pool, t_tmp_stream) : cudaMalloc(&p, b);
    if (e == cudaErrorMemoryAllocation && c) {  // give back what the pools keep and try again
        cudaGetLastError();
        cudaStreamSynchronize(pooled ? t_tmp_stream : c->stream);
        {
            std::lock_guard<std::mutex> lk(g_pools_mu);
            for (Ctx* o : g_pools)
                if (o->device == c->device) cudaMemPoolTrimTo(o->pool, 0);
        }
        e = pooled ? cudaMallocFromPoolAsync(&p, b, c->pool, t_tmp_stream) : cudaMalloc(&p, b);
    }
    if (e == cudaSuccess && pooled) stream = t_tmp_stream;
    if (e != cudaSuccess) {
        p = nullptr;
        if (c) c->allocated.fetch_sub((int64_t)b);
        cudaGetLastError();
        throw Error{VIE_ERR_OOM, "cudaMalloc of " + std::to_string(b) + " bytes failed: " + cudaGetErrorString(e),
                    e == cudaErrorMemoryAllocation};
    }
    bytes = b;
    owner = c;
    if (c) {
        int64_t pk = c->peak.load(), cur = c->allocated.load() + kept;
        while (cur > pk && !c->peak.compare_exchange_weak(pk, cur)) {
        }
    }
}

void DevBuf::release() {
    if (p) {
        if (stream) cudaFreeAsync(p, stream);
        else cudaFree(p);
        if (owner) owner->allocated.fetch_sub((int64_t)bytes);
    }
    p = nullptr;
    bytes = 0;
    owner = nullptr;
    stream = nullptr;
}

// ---------------------------------------------------------------------------
// Sec. 3 basis on a voxelised cube: one rooftop per voxel face.  Faces are
// numbered x-faces, y-faces, z-faces; inside a direction lexicographically in
// (i, j, k) with the normal index running 0..nv.
// ---------------------------------------------------------------------------
MeshTables build_mesh(double side, int nv) {
    MeshTables m;
    m.nv = nv;
    m.side = side;
    m.h = side / nv;
    m.nvox = nv * nv * nv;
    auto vnum = [nv](int i, int j, int k) { return (i * nv + j) * nv + k; };
    for (int i = 0; i < nv; ++i)
        for (int j = 0; j < nv; ++j)
            for (int k = 0; k < nv; ++k) {
                m.vox_ijk.push_back(i);
                m.vox_ijk.push_back(j);
                m.vox_ijk.push_back(k);
            }
    for (int d = 0; d < 3; ++d) {
        int ext[3] = {nv, nv, nv};
        ext[d] = nv + 1;
        for (int i = 0; i < ext[0]; ++i)
            for (int j = 0; j < ext[1]; ++j)
                for (int k = 0; k < ext[2]; ++k) {
                    int ijk[3] = {i, j, k};
                    int mm = ijk[d];
                    int f = (int)m.face_dir.size();
                    m.face_dir.push_back(d);
                    int below[3] = {i, j, k};
                    below[d] = mm - 1;
                    m.face_lo.push_back(mm >= 1 ? vnum(below[0], below[1], below[2]) : -1);
                    m.face_hi.push_back(mm <= nv - 1 ? vnum(i, j, k) : -1);
                    if (mm == 0 || mm == nv) {
                        m.face_sheet.push_back((int)m.surf_face.size());
                        m.face_sheet_sign.push_back(mm == 0 ? +1 : -1);
                        m.surf_face.push_back(f);
                    } else {
                        m.face_sheet.push_back(-1);
                        m.face_sheet_sign.push_back(0);
                    }
                }
    }
    m.np = (int)m.face_dir.size();
    m.nsurf = (int)m.surf_face.size();
    return m;
}

// ---------------------------------------------------------------------------
// Grid hierarchy (Sec. 5.1 Definition, Sec. 5.3 eq. eq_rec01, Sec. 5.4).
// Power-of-two quadtree over a root square of side s 2^L whose finest boxes
// (side s = smallest infinity-norm centre separation) hold at most one atom.
// Blocks are listed by level, then target box (y, x), then source box (y, x).
// ---------------------------------------------------------------------------
void build_tree(Op& op) {
    const int N = op.N;
    op.blocks.clear();
    op.block_atoms.clear();
    if (N == 1) {
        op.L = 0;
        return;
    }
    std::vector<double> x(N), y(N);
    for (int a = 0; a < N; ++a) {
        x[a] = op.centres[3 * a];
        y[a] = op.centres[3 * a + 1];
    }
    double s = std::numeric_limits<double>::infinity();
    for (int a = 0; a < N; ++a)
        for (int b = a + 1; b < N; ++b) s = std::min(s, std::max(std::fabs(x[a] - x[b]), std::fabs(y[a] - y[b])));
    if (!(s > 0)) fail(VIE_ERR_INVALID_ARG, "two atoms share the same (x, y) position");
    double xmin = *std::min_element(x.begin(), x.end()), xmax = *std::max_element(x.begin(), x.end());
    double ymin = *std::min_element(y.begin(), y.end()), ymax = *std::max_element(y.begin(), y.end());
    double ext = std::max(xmax - xmin, ymax - ymin);
    int L = 0;
    while (std::ldexp(1.0, L) < ext / s + 1.0 - 1e-9) ++L;
    if (L > 20) fail(VIE_ERR_INVALID_ARG, "atom layout needs more than 20 grid levels");
    op.L = L;
    const long long side_boxes = 1LL << L;
    std::vector<long long> fx(N), fy(N);
    for (int a = 0; a < N; ++a) {
        fx[a] = std::min(side_boxes - 1, std::max(0LL, (long long)std::floor((x[a] - (xmin - 0.5 * s)) / s)));
        fy[a] = std::min(side_boxes - 1, std::max(0LL, (long long)std::floor((y[a] - (ymin - 0.5 * s)) / s)));
    }
    for (int lev = 1; lev <= L; ++lev) {
        int shift = L - lev;
        std::map<std::pair<long long, long long>, std::vector<int>> boxes;  // key (y, x), sorted
        for (int a = 0; a < N; ++a) boxes[{fy[a] >> shift, fx[a] >> shift}].push_back(a);
        for (auto& tb : boxes) {
            long long ty = tb.first.first, tx = tb.first.second;
            // candidate source boxes: children of the 3x3 parent neighbourhood
            std::vector<std::pair<long long, long long>> cand;
            for (long long py = (ty >> 1) - 1; py <= (ty >> 1) + 1; ++py)
                for (long long px = (tx >> 1) - 1; px <= (tx >> 1) + 1; ++px)
                    for (int cy = 0; cy < 2; ++cy)
                        for (int cx = 0; cx < 2; ++cx) {
                            std::pair<long long, long long> key{2 * py + cy, 2 * px + cx};
                            if (py >= 0 && px >= 0 && boxes.count(key)) cand.push_back(key);
                        }
            std::sort(cand.begin(), cand.end());
            for (auto& key : cand) {
                long long dist = std::max(std::llabs(key.first - ty), std::llabs(key.second - tx));
                bool far = (lev == L) ? (dist != 0) : (dist > 1);
                if (!far) continue;
                const auto& ta = tb.second;
                const auto& sa = boxes[key];
                FarBlock b;
                b.level = lev;
                b.nt = (int)ta.size();
                b.ns = (int)sa.size();
                b.t_off = (int)op.block_atoms.size();
                op.block_atoms.insert(op.block_atoms.end(), ta.begin(), ta.end());
                b.s_off = (int)op.block_atoms.size();
                op.block_atoms.insert(op.block_atoms.end(), sa.begin(), sa.end());
                b.m = b.nt * op.np;
                b.n = b.ns * op.np;
                b.dist = (int)dist;
                b.dmin = (int)std::min(std::llabs(key.first - ty), std::llabs(key.second - tx));
                op.blocks.push_back(b);
            }
        }
    }
    // pair every block with its mirror (the far relation is symmetric)
    std::map<std::tuple<int, int, int>, int> idx;
    for (size_t i = 0; i < op.blocks.size(); ++i) {
        const auto& b = op.blocks[i];
        idx[{b.level, op.block_atoms[b.t_off], op.block_atoms[b.s_off]}] = (int)i;
    }
    for (size_t i = 0; i < op.blocks.size(); ++i) {
        auto& b = op.blocks[i];
        auto it = idx.find({b.level, op.block_atoms[b.s_off], op.block_atoms[b.t_off]});
        if (it == idx.end()) fail(VIE_ERR_STATE, "far block without a mirror");
        b.mirror = it->second;
    }
}

// ---------------------------------------------------------------------------
// App. C: greedy least-loaded assignment.  Interactions sorted by decreasing
// weight are given one by one to the currently least-loaded process (lowest
// index on ties).
// ---------------------------------------------------------------------------
void lpt_assign(const std::vector<double>& w, int nproc, std::vector<int>& owner, std::vector<double>& loads) {
    std::vector<int> order(w.size());
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return w[a] > w[b]; });
    using E = std::pair<double, int>;
    std::priority_queue<E, std::vector<E>, std::greater<E>> heap;
    for (int k = 0; k < nproc; ++k) heap.push({0.0, k});
    owner.assign(w.size(), 0);
    loads.assign(nproc, 0.0);
    for (int i : order) {
        E top = heap.top();
        heap.pop();
        owner[i] = top.second;
        loads[top.second] += w[i];
        heap.push({loads[top.second], top.second});
    }
}

// ---------------------------------------------------------------------------
// Work lists of the compressed apply (see apply.cu for the item layouts).
//  phase 1 (t = R x): item (block, k0, k1): rows k0..k1 of R_b
//  phase 2 (F = sum Q t): item (atom, p0, p1): rows p0..p1 of that atom,
//          looping over the blocks whose target box holds the atom
// Items are mapped to persistent CTAs with the greedy least-loaded rule,
// weighted by their factor bytes.
// ---------------------------------------------------------------------------
static void pack_lpt(const std::vector<int4>& items, const std::vector<double>& w, int ncta,
                     std::vector<int4>& out_items, std::vector<int>& cta_ptr, std::vector<int>* perm = nullptr,
                     const std::vector<uint64_t>* key = nullptr, double* most = nullptr) {
    std::vector<int> owner;
    std::vector<double> loads;
    lpt_assign(w, ncta, owner, loads);
    if (most) *most = *std::max_element(loads.begin(), loads.end());
    std::vector<std::vector<int>> per(ncta);
    // within a CTA keep the heaviest items first, or, given a spatial key, the
    // items in key order: every CTA then sweeps the array in the same
    // direction at about the same pace (its items' weights are spread evenly
    // over the keys), so the vector rows the CTAs gather at any one time come
    // from one region and stay in L2 (the order inside a CTA does not change
    // its load)
    std::vector<int> order(items.size());
    std::iota(order.begin(), order.end(), 0);
    if (key)
        std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return (*key)[a] < (*key)[b]; });
    else
        std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return w[a] > w[b]; });
    for (int i : order) per[owner[i]].push_back(i);
    out_items.clear();
    cta_ptr.assign(ncta + 1, 0);
    if (perm) perm->clear();
    for (int c = 0; c < ncta; ++c) {
        for (int i : per[c]) {
            out_items.push_back(items[i]);
            if (perm) perm->push_back(i);
        }
        cta_ptr[c + 1] = (int)out_items.size();
    }
}

// Load of one tensor-core tile in K stages: every stage moves the same bytes
// (A planes padded to 128 rows) and takes the same MMAs whatever the tile's
// real row count, so the rows do not enter; a tile also pays its accumulator
// drain, about two stages.
static double tile_cost(int64_t K, int ks) { return (double)((K + ks - 1) / ks) + 2.0; }

// Z-order (Morton) code of every atom centre, from its x, y position in the
// array's bounding box quantised to 16 bits per axis
static std::vector<uint64_t> atom_zorder(const Op& op) {
    // (a joined operator of several problems keeps no centres: one key for all)
    if (op.centres.size() < 3 * (size_t)op.N) return std::vector<uint64_t>(op.N, 0);
    double lo[2] = {std::numeric_limits<double>::max(), std::numeric_limits<double>::max()};
    double hi[2] = {-lo[0], -lo[1]};
    for (int a = 0; a < op.N; ++a)
        for (int d = 0; d < 2; ++d) {
            lo[d] = std::min(lo[d], op.centres[3 * a + d]);
            hi[d] = std::max(hi[d], op.centres[3 * a + d]);
        }
    std::vector<uint64_t> z(op.N);
    for (int a = 0; a < op.N; ++a) {
        uint32_t q[2];
        for (int d = 0; d < 2; ++d) {
            const double span = hi[d] - lo[d];
            const double f = span > 0 ? (op.centres[3 * a + d] - lo[d]) / span : 0.0;
            q[d] = (uint32_t)std::min(65535.0, std::max(0.0, std::floor(f * 65535.0 + 0.5)));
        }
        uint64_t code = 0;
        for (int bit = 15; bit >= 0; --bit) code = (code << 2) | (((q[1] >> bit) & 1u) << 1) | ((q[0] >> bit) & 1u);
        z[a] = code;
    }
    return z;
}

void build_apply_lists(Op& op) {
    const int nb = (int)op.blocks.size();
    std::vector<FarBlockDev> hb(std::max(nb, 1));
    int64_t toff = 0;
    for (int i = 0; i < nb; ++i) {
        auto& b = op.blocks[i];
        b.t_off_vec = toff;
        toff += b.rank;
        const int prob = op.block_prob.empty() ? 0 : op.block_prob[i];
        hb[i] = FarBlockDev{b.m, b.n, b.rank, b.nt, b.ns, b.t_off, b.s_off, prob, (long long)b.q_off,
                            (long long)b.rh_off, (long long)b.t_off_vec};
    }
    op.t_total = toff;
    upload(op.d_blocks, hb);
    upload(op.d_block_atoms, op.block_atoms.empty() ? std::vector<int>{0} : op.block_atoms);
    op.n_cta = op.ctx->n_sm * 3;

    // phase 1
    std::vector<int4> it1;
    std::vector<double> w1;
    // one item = up to 32 rows of R_b (8 warps x 4 rows); smaller blocks keep
    // whole rows together so that every warp of the CTA has work
    for (int i = 0; i < nb; ++i) {
        const auto& b = op.blocks[i];
        if (b.rank == 0) continue;
        int rc = 32;
        for (int k0 = 0; k0 < b.rank; k0 += rc) {
            int k1 = std::min(b.rank, k0 + rc);
            it1.push_back(make_int4(i, k0, k1, op.block_prob.empty() ? 0 : op.block_prob[i]));
            w1.push_back((double)(k1 - k0) * b.n);
        }
    }
    std::vector<int4> p1;
    std::vector<int> c1;
    pack_lpt(it1, w1, op.n_cta, p1, c1);
    op.n_p1_items = (int)p1.size();
    upload(op.d_p1_items, p1.empty() ? std::vector<int4>{make_int4(0, 0, 0, 0)} : p1);
    upload(op.d_p1_cta, c1);
    // the same items on two CTAs per SM: the multi-RHS kernels hold two CTAs
    // per SM (their register use), and a third list entry per SM would run as
    // a second wave
    op.n_cta_m = op.ctx->n_sm * 2;
    {
        std::vector<int4> q;
        std::vector<int> c;
        pack_lpt(it1, w1, op.n_cta_m, q, c);
        upload(op.d_p1m_items, q.empty() ? std::vector<int4>{make_int4(0, 0, 0, 0)} : q);
        upload(op.d_p1m_cta, c);
    }

    // phase 2: per atom the (block, slot) entries, then row chunks
    std::vector<std::vector<int2>> ent(op.N);
    for (int i = 0; i < nb; ++i) {
        const auto& b = op.blocks[i];
        if (b.rank == 0) continue;
        for (int s = 0; s < b.nt; ++s) ent[op.block_atoms[b.t_off + s]].push_back(make_int2(i, s));
    }
    std::vector<int> csr(op.N + 1, 0);
    std::vector<int2> flat;
    std::vector<double> rsum(op.N, 0.0);
    for (int a = 0; a < op.N; ++a) {
        for (auto e : ent[a]) {
            flat.push_back(e);
            rsum[a] += op.blocks[e.x].rank;
        }
        csr[a + 1] = (int)flat.size();
    }
    std::vector<int4> it2;
    std::vector<double> w2;
    const int rows_per_item = 128;
    for (int a = 0; a < op.N; ++a)
        for (int p0 = 0; p0 < op.np; p0 += rows_per_item) {
            int p1e = std::min(op.np, p0 + rows_per_item);
            it2.push_back(make_int4(a, p0, p1e, op.atom_prob.empty() ? 0 : op.atom_prob[a]));
            w2.push_back((double)(p1e - p0) * (rsum[a] + 1.0));
        }
    std::vector<int4> p2;
    std::vector<int> c2;
    pack_lpt(it2, w2, op.n_cta, p2, c2);
    op.n_p2_items = (int)p2.size();
    upload(op.d_p2_items, p2);
    upload(op.d_p2_cta, c2);
    {
        std::vector<int4> q;
        std::vector<int> c;
        pack_lpt(it2, w2, op.n_cta_m, q, c);
        upload(op.d_p2m_items, q);
        upload(op.d_p2m_cta, c);
    }

    // tensor-core path: 64-row output tiles (rows of R_b, rows of an atom)
    op.n_cta_tc = op.ctx->n_sm * 4;
    std::vector<int4> t1, t2;
    std::vector<double> wt1, wt2;
    for (int i = 0; i < nb; ++i) {
        const auto& b = op.blocks[i];
        for (int k0 = 0; k0 < b.rank; k0 += 64) {
            t1.push_back(make_int4(i, k0, std::min(b.rank, k0 + 64), 0));
            wt1.push_back(64.0 * b.n);
        }
    }
    for (int a = 0; a < op.N; ++a)
        for (int p0 = 0; p0 < op.np; p0 += 64) {
            t2.push_back(make_int4(a, p0, std::min(op.np, p0 + 64), 0));
            wt2.push_back(64.0 * (rsum[a] + 1.0));
        }
    std::vector<int4> q1, q2;
    std::vector<int> e1, e2;
    pack_lpt(t1, wt1, op.n_cta_tc, q1, e1);
    pack_lpt(t2, wt2, op.n_cta_tc, q2, e2);
    op.n_t1_items = (int)q1.size();
    op.n_t2_items = (int)q2.size();
    upload(op.d_t1_items, q1.empty() ? std::vector<int4>{make_int4(0, 0, 0, 0)} : q1);
    upload(op.d_t1_cta, e1);
    upload(op.d_t2_items, q2);
    upload(op.d_t2_cta, e2);
    upload(op.d_p2_csr, csr);
    upload(op.d_p2_ent, flat.empty() ? std::vector<int2>{make_int2(0, 0)} : flat);
    op.umma_ready = false;
    op.ws_ready = op.ws_packed = op.ws_pack_failed = false;
    op.d_ws_r.release();
    op.d_ws_q.release();

    // register-tile path: classes of blocks with the same factor storage, in
    // groups of up to kTileMembers members; phase 1 items of up to rows1 rows and
    // tile_seg columns of R, phase 2 items of up to rows2 rows of Q.  Rows are cut
    // into equal pieces (96 = 48 + 48), in storage order: the coarse levels'
    // long items come first.
    {
        std::map<std::pair<long long, int>, std::vector<int>> cls;
        double work = 0;  // complex products of phase 1
        for (int i = 0; i < nb; ++i) {
            const auto& b = op.blocks[i];
            if (b.rank == 0) continue;
            work += (double)b.rank * b.n;
            cls[{(long long)b.rh_off, op.block_prob.empty() ? 0 : op.block_prob[i]}].push_back(i);
        }
        // a segment of R (64 rows, 16 columns) is at most about a
        // sixteenth of an SM's share of the work, between 128 and 512 columns:
        // shorter ones on small operators, where one long item would be the last
        // to finish (12 x 12 array of 3^3 cubes in float64: 1.77 ms with 512)
        op.tile_seg = 128;
        while (op.tile_seg < 512 && 2.0 * op.tile_seg * 64 * 16 * 16 * op.ctx->n_sm <= work) op.tile_seg *= 2;
        const int seg_len = op.tile_seg;
        // Rows per item.  complex64: 64 of R and 256 of Q, or 32 and 64 where shared
        // factors leave an SM fewer than eight items of phase 1 (one column, us: 4 x 4
        // array of 3^3 cubes 36.0 -> 31.9, 8 x 8 70 -> 55, 16 x 16 153 -> 131; above, the
        // factor's staging counts: 20 x 20 222 -> 226, 28 x 28 of 4^3 763 -> 939; so it does
        // where no two blocks share: 35 atoms of the spiral, 3 columns, 64 -> 75).
        // complex128: 16 and 32 always; a product takes its SM's two float64 units
        // for so long that copies cost nothing and the last items' length everything
        // (8 x 8 array of 3^3 cubes, 1 column: 817 -> 447 us, 12 x 12, 3 columns: 2476 -> 2108).
        const bool wide = op.fprec == VIE_C128;
        int64_t nmem = 0, n64 = 0;
        for (const auto& kv : cls) {
            const auto& b = op.blocks[kv.second[0]];
            const int64_t cnt = (int64_t)kv.second.size();
            nmem += cnt;
            n64 += (cnt + kTileMembers - 1) / kTileMembers * ((b.n + seg_len - 1) / seg_len) *
                   ((b.rank + kTileRows1 - 1) / kTileRows1);
        }
        op.share_mean = cls.empty() ? 1.0 : (double)nmem / (double)cls.size();
        const bool fine = op.share_mean >= 3.0 && n64 < 8 * (int64_t)op.ctx->n_sm;
        const int rows1 = wide ? kTileRows1Wide : fine ? 32 : kTileRows1;
        const int rows2 = wide ? kTileRows2Wide : fine ? 64 : kTileRows2;
        std::vector<long long> poff(std::max(nb, 1), 0), ctoff(std::max(nb, 1), 0);
        std::vector<int> cseg;
        int64_t ptot = 0, ctot = 0;
        for (int i = 0; i < nb; ++i) {
            const auto& b = op.blocks[i];
            poff[i] = ptot;
            ctoff[i] = ctot;
            if (b.rank == 0) continue;
            ptot += (int64_t)b.nt * op.np;
            ctot += (int64_t)b.rank * ((b.n + seg_len - 1) / seg_len);
            if (b.n > seg_len) cseg.push_back(i);
        }
        std::vector<FarMember> cmem;
        std::vector<FarTile> c1, c2;
        op.tile_group = 1;
        for (const auto& kv : cls) {
            const auto& mem = kv.second;
            const auto& b = op.blocks[mem[0]];
            auto tiles = [](int rows, int most, auto&& f) {  // equal pieces of at most `most` rows
                const int nt = (rows + most - 1) / most;
                const int per = ((rows + nt - 1) / nt + 1) / 2 * 2;  // even: 16-byte copies
                for (int r0 = 0; r0 < rows; r0 += per) f(r0, std::min(per, rows - r0));
            };
            for (size_t g = 0; g < mem.size(); g += kTileMembers) {
                const int first = (int)cmem.size();
                const int cnt = (int)std::min<size_t>(kTileMembers, mem.size() - g);
                op.tile_group = std::max(op.tile_group, cnt);
                for (int j = 0; j < cnt; ++j) {
                    const int i = mem[g + j];
                    cmem.push_back(FarMember{ctoff[i], poff[i], op.blocks[i].s_off, 0});
                }
                const int prob = kv.first.second;
                for (int seg = 0; seg * seg_len < b.n; ++seg)
                    tiles(b.rank, rows1, [&](int r0, int rows) {
                        c1.push_back(FarTile{first, cnt, r0, rows, seg * seg_len, std::min(b.n, (seg + 1) * seg_len),
                                             seg, prob, b.rank, b.n, (long long)b.rh_off});
                    });
                tiles(b.m, rows2, [&](int r0, int rows) {
                    c2.push_back(FarTile{first, cnt, r0, rows, 0, 0, 0, prob, b.rank, b.m, (long long)b.q_off});
                });
            }
        }
        op.part_total = ptot;
        op.ct_total = ctot;
        op.n_c1_items = (int)c1.size();
        op.n_c2_items = (int)c2.size();
        upload(op.d_c1_items, c1.empty() ? std::vector<FarTile>{FarTile{}} : c1);
        upload(op.d_c2_items, c2.empty() ? std::vector<FarTile>{FarTile{}} : c2);
        // The same, longest first, for one or two columns of complex float32 on shared
        // factors and for complex128.  The storage order ends with the fine levels, whose
        // groups are the largest: with more items than resident CTAs these started last and set
        // the time (arrays of 3^3 cubes, 1 column, us: 7 x 7 70 -> 52, 11 x 11 119 -> 90, 28 x 28
        // 396 -> 369; complex128, 7 x 7, 471 -> 358).  With more columns, and in double-float,
        // an item is whole tiles whatever its class, and the storage order, in which
        // neighbours share x and factors, is up to 2% faster (16 x 16, 12 columns, 628 against
        // 635 us; double-float, 16 x 16 of 4^3, 1 column, 922 against 942); so it is without
        // shared factors (300 atoms of the spiral, 2 columns, 655 against 660).
        op.tile_long = wide || op.share_mean >= 3.0;
        if (!op.tile_long) c1.clear(), c2.clear();
        auto by_cost = [](std::vector<FarTile>& v, auto&& cost) {
            std::stable_sort(v.begin(), v.end(), [&](const FarTile& a, const FarTile& b) { return cost(a) > cost(b); });
        };
        by_cost(c1, [](const FarTile& t) { return (long long)(t.k1 - t.k0) * (8 + t.nm); });
        by_cost(c2, [](const FarTile& t) { return (long long)t.rank * (8 + t.nm); });
        upload(op.d_c1_long, c1.empty() ? std::vector<FarTile>{FarTile{}} : c1);
        upload(op.d_c2_long, c2.empty() ? std::vector<FarTile>{FarTile{}} : c2);
        op.n_cseg = (int)cseg.size();
        upload(op.d_cseg, cseg);
        upload(op.d_cmem, cmem.empty() ? std::vector<FarMember>{FarMember{}} : cmem);
        std::vector<long long> pbase;  // per entry of the atoms' (block, slot) lists
        for (const int2& e : flat) pbase.push_back(poff[e.x] + (long long)e.y * op.np);
        upload(op.d_pbase, pbase);
        upload(op.d_ctoff, ctoff);
        op.d_part.release();  // sized on first use (tile_reserve)
        op.d_ct.release();
        op.tile_oom = 0;
        op.tile_pinned = false;
    }
}

void build_umma_lists(Op& op) {
    if (op.umma_ready) return;
    const int nb = (int)op.blocks.size();
    constexpr int kRows = 128;
    op.n_cta_u = op.ctx->n_sm * 2;
    // phase 1: blocks with the same source atoms share x_J, so their R rows
    // are stacked into one tall operand and cut into 128-row tiles
    std::map<std::vector<int>, std::vector<int>> groups;
    for (int i = 0; i < nb; ++i) {
        const auto& b = op.blocks[i];
        if (b.rank == 0) continue;
        std::vector<int> key(op.block_atoms.begin() + b.s_off, op.block_atoms.begin() + b.s_off + b.ns);
        groups[key].push_back(i);
    }
    const std::vector<uint64_t> zc = atom_zorder(op);
    std::vector<long long> rowoff;
    std::vector<int> rowt;
    std::vector<int4> it1;
    std::vector<double> w1;
    std::vector<uint64_t> key1, key2;  // spatial keys: the source atoms' lowest Z-order code, the atom's
    for (const auto& kv : groups) {
        const int rep = kv.second.front();
        uint64_t zmin = ~0ull;
        for (int a : kv.first) zmin = std::min(zmin, zc[a]);
        const int64_t start = (int64_t)rowoff.size();
        for (int i : kv.second) {
            const auto& b = op.blocks[i];
            for (int k = 0; k < b.rank; ++k) {
                rowoff.push_back((long long)(b.rh_off + (int64_t)k * b.n));
                rowt.push_back((int)(b.t_off_vec + k));
            }
        }
        const int64_t total = (int64_t)rowoff.size() - start;
        for (int64_t r0 = 0; r0 < total; r0 += kRows) {
            const int nr = (int)std::min<int64_t>(kRows, total - r0);
            it1.push_back(make_int4(rep, (int)(start + r0), nr, op.block_prob.empty() ? 0 : op.block_prob[rep]));
            w1.push_back(tile_cost(op.blocks[rep].n, 32));
            key1.push_back(zmin);
        }
    }
    // phase 2: per atom every (block, rank index) as one virtual K axis
    std::vector<std::vector<int2>> ent(op.N);
    for (int i = 0; i < nb; ++i) {
        const auto& b = op.blocks[i];
        if (b.rank == 0) continue;
        for (int s = 0; s < b.nt; ++s) ent[op.block_atoms[b.t_off + s]].push_back(make_int2(i, s));
    }
    std::vector<long long> qoff, kptr(op.N + 1, 0);
    std::vector<int> tidx;
    std::vector<int4> it2;
    std::vector<double> w2;
    for (int a = 0; a < op.N; ++a) {
        for (auto e : ent[a]) {
            const auto& b = op.blocks[e.x];
            for (int k = 0; k < b.rank; ++k) {
                qoff.push_back((long long)(b.q_off + (int64_t)e.y * op.np + (int64_t)k * b.m));
                tidx.push_back((int)(b.t_off_vec + k));
            }
        }
        kptr[a + 1] = (long long)qoff.size();
        const double K = (double)(kptr[a + 1] - kptr[a]);
        for (int p0 = 0; p0 < op.np; p0 += kRows) {
            const int p1 = std::min(op.np, p0 + kRows);
            it2.push_back(make_int4(a, p0, p1, op.atom_prob.empty() ? 0 : op.atom_prob[a]));
            w2.push_back(tile_cost((int64_t)K, 32));
            key2.push_back(zc[a]);
        }
    }
    std::vector<int4> q1, q2;
    std::vector<int> e1, e2, p1, p2;
    pack_lpt(it1, w1, op.n_cta_u, q1, e1, &p1, &key1);
    pack_lpt(it2, w2, op.n_cta_u, q2, e2, &p2, &key2);
    op.n_u1_items = (int)q1.size();
    op.n_u2_items = (int)q2.size();
    upload(op.d_u1_rowoff, rowoff.empty() ? std::vector<long long>{0} : rowoff);
    upload(op.d_u1_rowt, rowt.empty() ? std::vector<int>{0} : rowt);
    upload(op.d_u1_items, q1.empty() ? std::vector<int4>{make_int4(0, 0, 0, 0)} : q1);
    upload(op.d_u1_cta, e1);
    upload(op.d_u2_qoff, qoff.empty() ? std::vector<long long>{0} : qoff);
    upload(op.d_u2_tidx, tidx.empty() ? std::vector<int>{0} : tidx);
    upload(op.d_u2_kptr, kptr);
    upload(op.d_u2_items, q2.empty() ? std::vector<int4>{make_int4(0, 0, 0, 0)} : q2);
    upload(op.d_u2_cta, e2);
    // packed variant: every item's A operand as whole 32-wide K stages, item
    // after item in work-list order; offsets in stages
    auto stage_offsets = [](const std::vector<int4>& items, auto nk_of, std::vector<long long>& off) {
        off.assign(items.size() + 1, 0);
        for (size_t i = 0; i < items.size(); ++i) off[i + 1] = off[i] + (nk_of(items[i]) + 31) / 32;
    };
    std::vector<long long> pk1, pk2;
    stage_offsets(q1, [&](const int4& it) { return (long long)op.blocks[it.x].n; }, pk1);
    stage_offsets(q2, [&](const int4& it) { return kptr[it.x + 1] - kptr[it.x]; }, pk2);
    op.u1_stages = pk1.back();
    op.u2_stages = pk2.back();
    upload(op.d_u1_pk, pk1);
    upload(op.d_u2_pk, pk2);
    op.umma_packed = false;
    op.umma_pack_failed = false;
    op.d_u1_pack.release();
    op.d_u2_pack.release();
    op.umma_ready = true;
}

// Lists of the warp-specialised kernels (apply_ws.cu has the plane layouts).
void build_ws_lists(Op& op) {
    if (op.ws_ready) return;
    const int nb = (int)op.blocks.size();
    const int nrt = (op.np + 127) / 128, n_cta = op.ctx->n_sm;
    const int per = (op.np + 7) / 8;  // chunks of 8 unknowns per atom (K axis of phase 1)
    // factor storages and where their planes lie
    std::vector<WsClass> cls;
    std::vector<int> cls_of(nb, -1), t0(nb, 0);
    std::unordered_map<long long, int> at;
    op.ws_r_units = op.ws_q_chunks = op.ws_t_total = 0;
    for (int i = 0; i < nb; ++i) {
        const auto& b = op.blocks[i];
        if (b.rank == 0) continue;
        const int G = (b.rank + 7) / 8;
        t0[i] = (int)(op.ws_t_total / 8);  // in units of 8 entries
        op.ws_t_total += 8 * G;
        const auto ins = at.emplace((long long)b.rh_off, (int)cls.size());
        if (ins.second) {
            cls.push_back(WsClass{(long long)b.rh_off, (long long)b.q_off, op.ws_r_units, op.ws_q_chunks, b.rank, b.n,
                                  b.m, 0});
            op.ws_r_units += (int64_t)((b.ns * per + 1) / 2) * G;
            op.ws_q_chunks += (int64_t)b.nt * G;
        }
        cls_of[i] = ins.first->second;
    }
    if (op.ws_t_total > std::numeric_limits<int>::max() || op.ws_q_chunks > std::numeric_limits<int>::max())
        fail(VIE_ERR_STATE, "the operator is too large for the warp-specialised apply's 32-bit places");
    op.ws_ncls = (int)cls.size();
    upload(op.d_ws_cls, cls.empty() ? std::vector<WsClass>{WsClass{}} : cls);
    const std::vector<uint64_t> zc = atom_zorder(op);
    // phase 1: blocks with the same source box (level and first source atom name
    // it) stack the 8-row groups of their R
    std::map<std::tuple<int, int, int>, std::vector<int>> groups;
    for (int i = 0; i < nb; ++i) {
        const auto& b = op.blocks[i];
        if (b.rank > 0) groups[{b.level, op.block_atoms[b.s_off], b.ns}].push_back(i);
    }
    std::vector<int> grp_t;
    struct Tile {
        int rep, grp0, ngrp, run0, nrun;
        uint64_t key;
    };
    std::vector<Tile> tiles;
    std::vector<WsRun> runs;
    for (const auto& kv : groups) {
        const int rep = kv.second.front();
        const FarBlock& rb = op.blocks[rep];
        uint64_t zmin = ~0ull;
        for (int s = 0; s < rb.ns; ++s) zmin = std::min(zmin, zc[op.block_atoms[rb.s_off + s]]);
        Tile T{rep, (int)grp_t.size(), 0, (int)runs.size(), 0, zmin};
        auto flush = [&] {
            if (T.ngrp == 0) return;
            grp_t.resize((size_t)T.grp0 + 16, 0);  // a tile's groups are 16 places apart
            tiles.push_back(T);
            T = Tile{rep, (int)grp_t.size(), 0, (int)runs.size(), 0, zmin};
        };
        for (int i : kv.second) {
            const WsClass& c = cls[cls_of[i]];
            const int G = (c.rank + 7) / 8;
            for (int g = 0; g < G;) {
                const int take = std::min(G - g, 16 - T.ngrp);
                runs.push_back(WsRun{c.r_unit + g, G, T.ngrp, take, 0});
                ++T.nrun;
                for (int e = 0; e < take; ++e) grp_t.push_back(t0[i] + g + e);
                T.ngrp += take;
                g += take;
                if (T.ngrp == 16) flush();
            }
        }
        flush();
    }
    upload(op.d_ws_grp, grp_t.empty() ? std::vector<int>{0} : grp_t);
    // phase 2: per atom the chunks of every (block, slot) touching it
    std::vector<int> cnt(op.N + 1, 0);
    for (int i = 0; i < nb; ++i) {
        const auto& b = op.blocks[i];
        if (b.rank == 0) continue;
        for (int s = 0; s < b.nt; ++s) cnt[op.block_atoms[b.t_off + s] + 1] += (b.rank + 7) / 8;
    }
    for (int a = 0; a < op.N; ++a) cnt[a + 1] += cnt[a];
    std::vector<int> fill(cnt.begin(), cnt.end() - 1), qidx(std::max(1, cnt[op.N])), tidx(std::max(1, cnt[op.N]));
    for (int i = 0; i < nb; ++i) {
        const auto& b = op.blocks[i];
        if (b.rank == 0) continue;
        const WsClass& c = cls[cls_of[i]];
        const int G = (c.rank + 7) / 8;
        for (int s = 0; s < b.nt; ++s) {
            int& f = fill[op.block_atoms[b.t_off + s]];
            for (int g = 0; g < G; ++g, ++f) {
                qidx[f] = (int)(c.q_chunk + (int64_t)s * G + g);
                tidx[f] = t0[i] + g;
            }
        }
    }
    upload(op.d_ws_kptr, cnt);
    upload(op.d_ws_qidx, qidx);
    upload(op.d_ws_tidx, tidx);
    // items per tile shape, mapped to one CTA per SM
    double load[2];  // the longest lists of the two phases, in K stages
    for (int v = 0; v < 2; ++v) {
        const int ks = v ? 16 : 32;
        std::vector<WsItem1> i1;
        std::vector<WsRun> rv;
        std::vector<double> w1;
        std::vector<uint64_t> k1;
        for (size_t i = 0; i < tiles.size(); ++i) {
            const Tile& A = tiles[i];
            const bool two = v && i + 1 < tiles.size() && tiles[i + 1].rep == A.rep;
            const Tile* Bt = two ? &tiles[i + 1] : nullptr;
            i1.push_back(WsItem1{A.rep, op.block_prob.empty() ? 0 : op.block_prob[A.rep], A.grp0, A.run0,
                                 {A.nrun, two ? Bt->nrun : 0}, {A.ngrp, two ? Bt->ngrp : 0}});
            w1.push_back(tile_cost(8ll * per * op.blocks[A.rep].ns, ks));
            k1.push_back(A.key);
            if (two) ++i;
        }
        std::vector<WsItem2> i2;
        std::vector<double> w2;
        std::vector<uint64_t> k2;
        for (int a = 0; a < op.N; ++a)
            for (int rt = 0; rt < nrt; rt += v + 1) {
                auto rows = [&](int t) { return std::max(0, std::min(128, op.np - t * 128)); };
                const int prob = op.atom_prob.empty() ? 0 : op.atom_prob[a];
                i2.push_back(WsItem2{a, prob, rt, {rows(rt), v ? rows(rt + 1) : 0}});
                w2.push_back(tile_cost(8ll * (cnt[a + 1] - cnt[a]), ks));
                k2.push_back(zc[a]);
            }
        auto place = [&](auto& items, const std::vector<double>& w, const std::vector<uint64_t>& key, DevBuf& d_items,
                         DevBuf& d_cta) -> double {
            using I = typename std::decay_t<decltype(items)>::value_type;
            std::vector<int4> dummy(items.size(), make_int4(0, 0, 0, 0)), out;
            std::vector<int> cta, perm;
            double most = 0.0;
            pack_lpt(dummy, w, n_cta, out, cta, &perm, &key, &most);
            std::vector<I> sorted(std::max<size_t>(1, items.size()));
            for (size_t i = 0; i < perm.size(); ++i) sorted[i] = items[perm[i]];
            upload(d_items, sorted);
            upload(d_cta, cta);
            return most;
        };
        op.n_ws1[v] = (int)i1.size();
        load[v] = place(i1, w1, k1, op.d_ws1_items[v], op.d_ws1_cta[v]) +
                  place(i2, w2, k2, op.d_ws2_items[v], op.d_ws2_cta[v]);
        upload(op.d_ws_runs[v], runs.empty() ? std::vector<WsRun>{WsRun{}} : runs);
    }
    // Which of them up to 32 columns take (variant 9 or 10).  Two row tiles per B tile read
    // and split the B operand once for twice the rows, which makes balanced lists 6 to 12%
    // faster, but halve the items: an SM's longest list may grow.  They win up to 1.15
    // times the load (35 arrays of 240 to 756 unknowns per atom, 8 to 32 columns: within 2% of the
    // faster one; us at 16 columns: 16 x 16 of 4^3 cubes 484 with one, 439 with two, 18 x 18 655 and
    // 740, lens-graded 9 x 9 159 and 223).  Atoms of one row tile leave the second one empty in
    // phase 2: always one (500 atoms of 108 unknowns: 733 against 813 us at 16 columns, 835 against
    // 912 at 32).
    op.ws_tiles = nrt > 1 && load[1] <= 1.15 * load[0] ? 2 : 1;
    op.ws_ready = true;
}

}  // namespace vie
