// Plane waves and fields of the rooftop basis, in float64: the right-hand side
// b = j k v0 (paper Sec. 3, eq. matrixeq), the radiation vector behind the far
// field and the cross sections, and the scattered near field (Sec. 2, eq.
// IntEq).  All of them use the 3-point Gauss rule per voxel axis.
//
// A plane wave over a rooftop factorises over the axes.  With the atom's low
// corner o and voxel indices i, and with e_n(x) = exp(j k q_n x),
//   int w_f exp(j k q . r) dV = h exp(j k q . o) P_d(i_d) T_a(i_a) T_b(i_b),
//   T_n(i) = e_n(h i) s_n,                    s_n = sum_p w_p e_n(h x_p)
//   P_d(i) = e_d(h (i-1)) a_d + e_d(h i) b_d  (a: weight x_p, b: weight 1 - x_p;
//                                              a term without its voxel is zero)
// so per direction one value per face of each atom type (`V`) and one phase per
// atom (`ph`) stand for the 27 or 54 exponentials per unknown of the written-out
// sum, and the unknowns cost one complex product each.
#include <algorithm>
#include <cmath>

#include "common.h"
#include "cplx.cuh"

namespace vie {

namespace {

// Gauss-Legendre on [0, 1]
__constant__ double c_x3[3] = {0.11270166537925831148, 0.5, 0.88729833462074168852};
__constant__ double c_w3[3] = {5.0 / 18.0, 8.0 / 18.0, 5.0 / 18.0};

struct Geo {
    const double* centres;
    const int* types;
    const double* sides;
    int N, T, nv, np;
};
Geo geo_of(const Op& op) {
    return {op.d_centres.as<double>(), op.d_types.as<int>(), op.d_sides.as<double>(), op.N, op.T, op.mesh.nv, op.np};
}

// rooftop face numbering of an atom (x-faces, then y, then z; each direction
// lexicographic in (i, j, k) with the normal index 0..nv)
__device__ __forceinline__ int face_index(int nv, int d, int i, int j, int k) {
    const int base = d * nv * nv * (nv + 1);
    if (d == 0) return base + (i * nv + j) * nv + k;
    if (d == 1) return base + (i * (nv + 1) + j) * nv + k;
    return base + (i * nv + j) * (nv + 1) + k;
}

__device__ __forceinline__ double2 cis(double ph) {
    double s, c;
    sincos(ph, &s, &c);
    return make_double2(c, s);
}

// ---------------------------------------------------------------------------
// Tables of W plane waves exp(j sign k q . r), q = vec + 3 w:
//   V[(t W + w) np + f] and ph[w N + a]; with `pol` (the right-hand side) V
//   carries the factor j k pol_d.
// blockIdx.y < T: the face values of one type; the rest: phases of 256 atoms.
// A few thousand exponentials in all, so latency bound.
// ---------------------------------------------------------------------------
constexpr int kMaxNv = 16;
__global__ void __launch_bounds__(256) k_pw_tables(Geo g, const double* __restrict__ vec, double sign, double k,
                                                   const double* __restrict__ pol, int W, double2* __restrict__ V,
                                                   double2* __restrict__ ph) {
    const int w = blockIdx.x;
    const double q[3] = {sign * vec[3 * w], sign * vec[3 * w + 1], sign * vec[3 * w + 2]};
    if ((int)blockIdx.y >= g.T) {
        const int a = ((int)blockIdx.y - g.T) * 256 + threadIdx.x;
        if (a >= g.N) return;
        const double hs = 0.5 * g.sides[g.types[a]];
        ph[(size_t)w * g.N + a] = cis(k * (q[0] * (g.centres[3 * a] - hs) + q[1] * (g.centres[3 * a + 1] - hs) +
                                           q[2] * (g.centres[3 * a + 2] - hs)));
        return;
    }
    const int t = blockIdx.y, nv = g.nv;
    const double h = g.sides[t] / nv;
    __shared__ double2 sE[3][3], sI[3][kMaxNv], sT[3][kMaxNv], sP[3][kMaxNv + 1];
    const int tid = threadIdx.x;
    if (tid < 9) sE[tid / 3][tid % 3] = cis(k * q[tid / 3] * h * c_x3[tid % 3]);
    for (int e = tid; e < 3 * nv; e += 256) sI[e / nv][e % nv] = cis(k * q[e / nv] * h * (e % nv));
    __syncthreads();
    for (int e = tid; e < 3 * (nv + 1); e += 256) {
        const int n = e / (nv + 1), i = e % (nv + 1);
        double2 s = make_double2(0, 0), a = make_double2(0, 0), b = make_double2(0, 0);
        for (int p = 0; p < 3; ++p) {
            s += c_w3[p] * sE[n][p];
            a += (c_w3[p] * c_x3[p]) * sE[n][p];
            b += (c_w3[p] * (1.0 - c_x3[p])) * sE[n][p];
        }
        double2 P = make_double2(0, 0);
        if (i >= 1) P += cmul(sI[n][i - 1], a);
        if (i < nv) {
            P += cmul(sI[n][i], b);
            sT[n][i] = cmul(sI[n][i], s);
        }
        if (pol) {  // j k pol_n
            const double2 jp = make_double2(-k * pol[6 * w + 2 * n + 1], k * pol[6 * w + 2 * n]);
            P = cmul(jp, P);
        }
        sP[n][i] = h * P;
    }
    __syncthreads();
    double2* out = V + ((size_t)t * W + w) * g.np;
    const int per = nv * nv * (nv + 1);
    for (int f = tid; f < g.np; f += 256) {
        const int d = f / per, r = f - d * per;
        const int n2 = d == 2 ? nv + 1 : nv, n1 = d == 1 ? nv + 1 : nv;
        const int i2 = r % n2, i1 = (r / n2) % n1, i0 = r / (n2 * n1);
        const double2 x = d == 0 ? sP[0][i0] : sT[0][i0];
        const double2 y = d == 1 ? sP[1][i1] : sT[1][i1];
        const double2 z = d == 2 ? sP[2][i2] : sT[2][i2];
        out[f] = cmul(cmul(x, y), z);
    }
}

// b[row, w] = ph V, one column per blockIdx.y.  Bound by the float64 units (one
// complex product per unknown) with the stores close behind.
__global__ void __launch_bounds__(256) k_pw_rhs(Geo g, const double2* __restrict__ V, const double2* __restrict__ ph,
                                                int W, double2* __restrict__ b, int64_t ld) {
    const int w = blockIdx.y;
    const unsigned n = (unsigned)g.N * g.np, np = g.np;
    double2* out = b + (int64_t)w * ld;
    for (unsigned r = blockIdx.x * 256 + threadIdx.x; r < n; r += gridDim.x * 256) {
        const unsigned a = r / np, f = r - a * np;
        out[r] = cmul(ph[(size_t)w * g.N + a], V[((size_t)g.types[a] * W + w) * np + f]);
    }
}

// ---------------------------------------------------------------------------
// Radiation vector N(q) = int J exp(j k q . r) dV: part[((z W + w) C + c) 3 + d]
// of the atoms of chunk z, for the columns c of blockIdx.z (kRC at a time; with
// `diag` only column w of direction w).  The factor ph V is formed once for
// the kRC columns, so an unknown costs one complex product per column and
// 1 / kRC for the factor: float64 bound.
// ---------------------------------------------------------------------------
constexpr int kRC = 4;

template <int K>
__device__ __forceinline__ void block_sum(double (&v)[K], double (*sh)[K]) {  // sh[8][K], result in v of thread 0..
#pragma unroll
    for (int i = 0; i < K; ++i)
        for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_down_sync(0xffffffffu, v[i], o);
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int i = 0; i < K; ++i) sh[threadIdx.x >> 5][i] = v[i];
    __syncthreads();
}

__global__ void __launch_bounds__(256) k_radiate(Geo g, const double2* __restrict__ V, const double2* __restrict__ ph,
                                                 int W, int w0, const double2* __restrict__ I, int C, int diag,
                                                 int atoms_per, int nz, double2* __restrict__ part) {
    const int w = blockIdx.x, z = blockIdx.y;
    const int c0 = diag ? w0 + w : blockIdx.z * kRC, nc = diag ? 1 : min(kRC, C - c0);
    const int a0 = z * atoms_per, na = min(atoms_per, g.N - a0);
    const int per = g.nv * g.nv * (g.nv + 1);
    const int64_t n = (int64_t)g.N * g.np;
    __shared__ double sh[8][6 * kRC];
    double acc[6 * kRC];
#pragma unroll
    for (int i = 0; i < 6 * kRC; ++i) acc[i] = 0.0;
#pragma unroll
    for (int d = 0; d < 3; ++d)
        for (int e = threadIdx.x; e < na * per; e += 256) {
            const int al = e / per, a = a0 + al, f = d * per + e - al * per;
            const double2 m = cmul(ph[(size_t)w * g.N + a], V[((size_t)g.types[a] * W + w) * g.np + f]);
            const double2* x = I + (int64_t)c0 * n + (int64_t)a * g.np + f;
#pragma unroll
            for (int c = 0; c < kRC; ++c)
                if (c < nc) {
                    const double2 v = x[(int64_t)c * n];
                    double& re = acc[(c * 3 + d) * 2];
                    double& im = acc[(c * 3 + d) * 2 + 1];
                    re = fma(m.x, v.x, re);
                    re = fma(-m.y, v.y, re);
                    im = fma(m.x, v.y, im);
                    im = fma(m.y, v.x, im);
                }
        }
    block_sum<6 * kRC>(acc, sh);
    if ((int)threadIdx.x < 3 * nc) {
        double2 s = make_double2(0, 0);
        for (int q = 0; q < 8; ++q) s += make_double2(sh[q][2 * threadIdx.x], sh[q][2 * threadIdx.x + 1]);
        const int c = threadIdx.x / 3, d = threadIdx.x % 3;
        const size_t col = diag ? 0 : c0 + c, cols = diag ? 1 : C;
        part[(((size_t)z * W + w) * cols + col) * 3 + d] = s;
    }
}

// F = -j k / (4 pi) (N - rhat (rhat . N)) for direction w0 + w, column c:
// out[(c npts + w0 + w) 3 + d]; or, with `pol` (diag), ext[w0 + w] =
// Re sum_d pol_d conj(N_d): the extinction Re(I^H v0), v0_i = int w_i . E0.
__global__ void k_far_finish(const double2* __restrict__ part, int W, int w0, int C, int nz,
                             const double* __restrict__ dirs, double k, int npts, double2* __restrict__ out,
                             const double* __restrict__ pol, double* __restrict__ ext) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= W * C) return;
    const int w = t / C, c = t % C;
    double2 N[3];
    for (int d = 0; d < 3; ++d) {
        N[d] = make_double2(0, 0);
        for (int z = 0; z < nz; ++z) N[d] += part[(((size_t)z * W + w) * C + c) * 3 + d];
    }
    if (pol) {
        double e = 0.0;
        for (int d = 0; d < 3; ++d) e += pol[6 * (w0 + w) + 2 * d] * N[d].x + pol[6 * (w0 + w) + 2 * d + 1] * N[d].y;
        ext[w0 + w] = e;
        return;
    }
    const double* r = dirs + 3 * (w0 + w);
    const double2 dot = r[0] * N[0] + r[1] * N[1] + r[2] * N[2];
    const double s = -k * 0.07957747154594766788;  // k / (4 pi)
    for (int d = 0; d < 3; ++d) {
        const double2 v = N[d] - r[d] * dot;
        out[((size_t)c * npts + w0 + w) * 3 + d] = make_double2(-s * v.y, s * v.x);
    }
}

// sca[c] = sum_p wt[p] |F(p, c)|^2
__global__ void __launch_bounds__(256) k_sphere_sum(const double2* __restrict__ F, const double* __restrict__ wt,
                                                    int npts, double* __restrict__ sca) {
    const double2* f = F + (size_t)blockIdx.x * npts * 3;
    __shared__ double sh[8][1];
    double v[1] = {0.0};
    for (int e = threadIdx.x; e < npts * 3; e += 256) v[0] += wt[e / 3] * (f[e].x * f[e].x + f[e].y * f[e].y);
    block_sum<1>(v, sh);
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int q = 0; q < 8; ++q) s += sh[q][0];
        sca[blockIdx.x] = s;
    }
}

// ---------------------------------------------------------------------------
// Scattered near field E = -j k A + (1 / (j k)) grad Phi at points outside the
// atoms, A = int J g, Phi = int q g (q = div J with the boundary sheets).
// One Gauss point costs one Green's function (square root, sine and cosine:
// ~60 float64 operations, the bound) whatever the number of columns: per voxel
// the sums S = sum w g, S_d = sum w x_d g and K = sum w grad g are formed, and a
// column takes them with its six face currents.  The sums over z run
// innermost, so a Gauss point adds to four sums instead of seven.
// part[((z npts + p) C + c) 3 + d], chunk z of the atoms, points of this pass.
// ---------------------------------------------------------------------------
struct GreenSum {
    double2 g, f;  // exp(-j k R) / R and (1 + j k R) g / R^2 (both times 4 pi, the sign of grad g apart)
};
__device__ __forceinline__ GreenSum green_pt(double r2, double k, double two_over_lambda) {
    const double inv = rsqrt(r2), R = r2 * inv;
    double sn, cs;
    sincospi(R * two_over_lambda, &sn, &cs);
    const double2 g = make_double2(cs * inv, -sn * inv);
    const double i2 = inv * inv, kr = k * R;
    return {g, make_double2(i2 * (g.x - kr * g.y), i2 * (g.y + kr * g.x))};
}
__device__ __forceinline__ void axpy(double2& a, double s, double2 x) {
    a.x = fma(s, x.x, a.x);
    a.y = fma(s, x.y, a.y);
}

__global__ void __launch_bounds__(256) k_near(DevMesh m, Geo geo, double k, const double2* __restrict__ I, int C,
                                              const double* __restrict__ pts, int npts, int atoms_per,
                                              double2* __restrict__ part) {
    const int ip = blockIdx.x, z = blockIdx.y, c0 = blockIdx.z * kRC, nc = min(kRC, C - c0);
    const int a0 = z * atoms_per, na = min(atoms_per, geo.N - a0);
    const double P[3] = {pts[3 * ip], pts[3 * ip + 1], pts[3 * ip + 2]};
    const double tol = k / 3.14159265358979323846, ik = 1.0 / k;
    const int nv = m.nv;
    const int64_t n = (int64_t)geo.N * m.np;
    const double2* Ic = I + (int64_t)c0 * n;
    __shared__ double sh[8][6 * kRC];
    double acc[6 * kRC];
#pragma unroll
    for (int i = 0; i < 6 * kRC; ++i) acc[i] = 0.0;
    // E_d += -j k A_d + K_d q / (j k), for grad g = -f (r - r') and A, K times 4 pi
    auto add = [&](int c, int d, double2 A, double2 K, double2 q) {
        const double2 kq = cmul(K, q);
        acc[(c * 3 + d) * 2] += k * A.y - ik * kq.y;
        acc[(c * 3 + d) * 2 + 1] += ik * kq.x - k * A.x;
    };
    for (int e = threadIdx.x; e < na * m.nvox; e += 256) {
        const int al = e / m.nvox, a = a0 + al, v = e - al * m.nvox;
        const double side = geo.sides[geo.types[a]], h = side / nv;
        const int vi[3] = {m.vox_ijk[3 * v], m.vox_ijk[3 * v + 1], m.vox_ijk[3 * v + 2]};
        double o[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) o[d] = P[d] - (geo.centres[3 * a + d] - 0.5 * side + h * vi[d]);
        double2 S = make_double2(0, 0), S3[3], K[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) S3[d] = K[d] = make_double2(0, 0);
        for (int ix = 0; ix < 3; ++ix) {
            const double dx = o[0] - h * c_x3[ix];
            double2 gx = make_double2(0, 0), fx = make_double2(0, 0);
            for (int iy = 0; iy < 3; ++iy) {
                const double dy = o[1] - h * c_x3[iy], r2 = dx * dx + dy * dy;
                double2 gy = make_double2(0, 0), fy = make_double2(0, 0), gz = make_double2(0, 0), fz = gz;
#pragma unroll
                for (int iz = 0; iz < 3; ++iz) {
                    const double dz = o[2] - h * c_x3[iz];
                    const GreenSum G = green_pt(fma(dz, dz, r2), k, tol);
                    axpy(gy, c_w3[iz], G.g);
                    axpy(gz, c_w3[iz] * c_x3[iz], G.g);
                    axpy(fy, c_w3[iz], G.f);
                    axpy(fz, c_w3[iz] * dz, G.f);
                }
                axpy(gx, c_w3[iy], gy);
                axpy(fx, c_w3[iy], fy);
                const double wxy = c_w3[ix] * c_w3[iy];
                axpy(S3[2], wxy, gz);
                axpy(K[2], wxy, fz);
                axpy(S3[1], wxy * c_x3[iy], gy);
                axpy(K[1], wxy * dy, fy);
            }
            axpy(S, c_w3[ix], gx);
            axpy(S3[0], c_w3[ix] * c_x3[ix], gx);
            axpy(K[0], c_w3[ix] * dx, fx);
        }
        // J = h^-2 (lo (1 - x) + up x) e_d, q = h^-3 sum (up - lo), dV = h^3
#pragma unroll
        for (int c = 0; c < kRC; ++c)
            if (c < nc) {
                const double2* Ia = Ic + (int64_t)c * n + (int64_t)a * m.np;
                double2 lo[3], up[3], q = make_double2(0, 0);
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    lo[d] = Ia[face_index(nv, d, vi[0], vi[1], vi[2])];
                    up[d] = Ia[face_index(nv, d, vi[0] + (d == 0), vi[1] + (d == 1), vi[2] + (d == 2))];
                    q += up[d] - lo[d];
                }
#pragma unroll
                for (int d = 0; d < 3; ++d) add(c, d, h * (cmul(lo[d], S - S3[d]) + cmul(up[d], S3[d])), K[d], q);
            }
    }
    for (int e = threadIdx.x; e < na * m.nsurf; e += 256) {
        const int al = e / m.nsurf, a = a0 + al, sf = e - al * m.nsurf;
        const double side = geo.sides[geo.types[a]], h = side / nv;
        const int f = m.surf_face[sf];
        const int4 fi = m.face[f];
        const int d0 = fi.x, v = fi.y >= 0 ? fi.y : fi.z;
        double o[3];
#pragma unroll
        for (int d = 0; d < 3; ++d)  // the face is the top of its lower voxel, or the bottom of its upper one
            o[d] = P[d] - (geo.centres[3 * a + d] - 0.5 * side + h * (m.vox_ijk[3 * v + d] + (d == d0 && fi.y >= 0)));
        double2 K[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) K[d] = make_double2(0, 0);
        for (int p = 0; p < 9; ++p) {
            const int i1 = p / 3, i2 = p - 3 * i1;
            double r[3];
#pragma unroll
            for (int d = 0; d < 3; ++d)  // in-plane axes in order: the first takes i1, the second i2
                r[d] = d == d0 ? o[d] : o[d] - h * c_x3[d == (d0 == 0 ? 1 : 0) ? i1 : i2];
            const GreenSum G = green_pt(r[0] * r[0] + r[1] * r[1] + r[2] * r[2], k, tol);
            const double w = c_w3[i1] * c_w3[i2];
#pragma unroll
            for (int d = 0; d < 3; ++d) axpy(K[d], w * r[d], G.f);
        }
        // density sign h^-2, dS = h^2
        const double sg = m.sheet_sign[f];
#pragma unroll
        for (int c = 0; c < kRC; ++c)
            if (c < nc) {
                const double2 q = sg * Ic[(int64_t)c * n + (int64_t)a * m.np + f];
#pragma unroll
                for (int d = 0; d < 3; ++d) add(c, d, make_double2(0, 0), K[d], q);
            }
    }
    block_sum<6 * kRC>(acc, sh);
    if ((int)threadIdx.x < 3 * nc) {
        double2 s = make_double2(0, 0);
        for (int q = 0; q < 8; ++q) s += make_double2(sh[q][2 * threadIdx.x], sh[q][2 * threadIdx.x + 1]);
        part[(((size_t)z * npts + ip) * C + c0 + threadIdx.x / 3) * 3 + threadIdx.x % 3] =
            0.07957747154594766788 * s;  // 1 / (4 pi)
    }
}

// points [p0, p0 + npts) of `total`
__global__ void k_near_finish(const double2* __restrict__ part, int npts, int C, int nz, int64_t p0, int64_t total,
                              double2* __restrict__ out) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= npts * C * 3) return;
    const int d = t % 3, c = (t / 3) % C, p = t / (3 * C);
    double2 s = make_double2(0, 0);
    for (int z = 0; z < nz; ++z) s += part[(((size_t)z * npts + p) * C + c) * 3 + d];
    out[(c * total + p0 + p) * 3 + d] = s;
}

// points or directions of one pass: a chunk of atoms' partial sums stay within 32 MB,
// and their number within 32 bits (as many sums as outputs in one pass would double
// what a call with many points holds)
int sum_cols(int nrhs, int npts) {
    return (int)std::max<int64_t>(1, std::min<int64_t>(npts, ((int64_t)32 << 20) / (48ll * nrhs)));
}

void grow(DevBuf& b, size_t bytes) {
    if (b.bytes < bytes) b.alloc(bytes);
}

// chunks of the atoms per output, so that `blocks` x chunks fill the GPU about
// four times over, with at least `min_atoms` atoms in a chunk (the partial sums of a
// chunk cost a block reduction)
int atom_chunks(const Op& op, int64_t blocks, int min_atoms) {
    const int64_t want = (4ll * op.ctx->n_sm + blocks - 1) / std::max<int64_t>(1, blocks);
    return (int)std::max<int64_t>(1, std::min<int64_t>({want, (int64_t)(op.N / min_atoms), (int64_t)64}));
}


// room in b for `want` columns of `per` bytes, or for as many as there is memory for
int fit(DevBuf& b, size_t per, int want) {
    while (b.bytes < per * want) {
        try {
            b.alloc(per * want);
        } catch (const Error& e) {
            if (!e.memory || want == 1) throw;
            want = (want + 1) / 2;
        }
    }
    return want;
}

// directions of one pass: their tables (op.d_pw) stay within 32 MB (or one direction's)
int table_cols(Op& op, int W) {
    const size_t per = ((size_t)op.T * op.np + op.N) * sizeof(double2);
    const size_t most = std::min<size_t>({(size_t)W, ((size_t)32 << 20) / per, (size_t)65535});
    return fit(op.d_pw, per, (int)std::max<size_t>(1, most));
}

double2* tables(Op& op, const double* vec, double sign, const double* pol, int W, double2** ph, cudaStream_t s) {
    const size_t nV = (size_t)op.T * W * op.np;
    double2* V = op.d_pw.as<double2>();
    *ph = V + nV;
    k_pw_tables<<<dim3(W, op.T + (op.N + 255) / 256), 256, 0, s>>>(geo_of(op), vec, sign, op.k, pol, W, V, *ph);
    VIE_CHECK_LAUNCH();
    return V;
}

}  // namespace

IncidentDev upload_incident(Op& op, const vie_incident* inc, int nrhs, cudaStream_t s) {
    grow(op.d_inc, (size_t)9 * nrhs * sizeof(double));
    double* d = op.d_inc.as<double>();
    // (a copy from pageable memory has read it when the call returns)
    VIE_CUDA(cudaMemcpyAsync(d, inc->khat, (size_t)3 * nrhs * sizeof(double), cudaMemcpyHostToDevice, s));
    VIE_CUDA(cudaMemcpyAsync(d + 3 * nrhs, inc->pol, (size_t)6 * nrhs * sizeof(double), cudaMemcpyHostToDevice, s));
    return {d, d + 3 * nrhs};
}

// b = j k v0, v0_i = int w_i . E0, E0 = pol exp(-j k khat . r)
void rhs_kernel_launch(Op& op, const double* d_khat, const double* d_pol, int nrhs, void* b, int64_t ld,
                       cudaStream_t s) {
    const int wc = table_cols(op, nrhs);
    const int64_t n = op.n();
    for (int w0 = 0; w0 < nrhs; w0 += wc) {
        const int W = std::min(wc, nrhs - w0);
        double2* ph;
        const double2* V = tables(op, d_khat + 3 * w0, -1.0, d_pol + 6 * w0, W, &ph, s);
        const int64_t bx = std::min<int64_t>((n + 255) / 256, std::max<int64_t>(1, 32ll * op.ctx->n_sm / W));
        k_pw_rhs<<<dim3((unsigned)bx, W), 256, 0, s>>>(geo_of(op), V, ph, W, (double2*)b + (int64_t)w0 * ld, ld);
        VIE_CHECK_LAUNCH();
    }
}

// far-field amplitudes of nrhs currents in npts directions: d_out[(c npts + p) 3 + d]
void far_field_launch(Op& op, const void* d_I, int nrhs, const double* d_dirs, int npts, void* d_out,
                      cudaStream_t s) {
    const int groups = (nrhs + kRC - 1) / kRC;
    int wc = table_cols(op, sum_cols(nrhs, npts));
    int nz = atom_chunks(op, (int64_t)wc * groups, 4);
    const int per = (op.N + nz - 1) / nz;
    nz = (op.N + per - 1) / per;
    wc = fit(op.d_fpart, (size_t)nz * nrhs * 3 * sizeof(double2), wc);
    for (int w0 = 0; w0 < npts; w0 += wc) {
        const int W = std::min(wc, npts - w0);
        double2* ph;
        const double2* V = tables(op, d_dirs + 3 * w0, 1.0, nullptr, W, &ph, s);
        k_radiate<<<dim3(W, nz, groups), 256, 0, s>>>(geo_of(op), V, ph, W, w0, (const double2*)d_I, nrhs, 0, per, nz,
                                                      op.d_fpart.as<double2>());
        VIE_CHECK_LAUNCH();
        k_far_finish<<<(W * nrhs + 127) / 128, 128, 0, s>>>(op.d_fpart.as<double2>(), W, w0, nrhs, nz, d_dirs, op.k,
                                                            npts, (double2*)d_out, nullptr, nullptr);
        VIE_CHECK_LAUNCH();
    }
}

// d_ext[c] = Re(I_c^H v0_c), the extinction: with v0 = int w . pol exp(-j k khat . r)
// it is Re sum_d pol_d conj(N_d(khat)) of the column's own radiation vector
void extinction_launch(Op& op, const void* d_I, const double* d_khat, const double* d_pol, int nrhs, double* d_ext,
                       cudaStream_t s) {
    const int wc = table_cols(op, nrhs);
    for (int w0 = 0; w0 < nrhs; w0 += wc) {
        const int W = std::min(wc, nrhs - w0);
        double2* ph;
        const double2* V = tables(op, d_khat + 3 * w0, 1.0, nullptr, W, &ph, s);
        int nz = atom_chunks(op, W, 4);
        const int per = (op.N + nz - 1) / nz;
        nz = (op.N + per - 1) / per;
        grow(op.d_fpart, (size_t)nz * W * 3 * sizeof(double2));
        k_radiate<<<dim3(W, nz, 1), 256, 0, s>>>(geo_of(op), V, ph, W, w0, (const double2*)d_I, nrhs, 1, per, nz,
                                                 op.d_fpart.as<double2>());
        VIE_CHECK_LAUNCH();
        k_far_finish<<<(W + 127) / 128, 128, 0, s>>>(op.d_fpart.as<double2>(), W, w0, 1, nz, nullptr, op.k, nrhs,
                                                     nullptr, d_pol, d_ext);
        VIE_CHECK_LAUNCH();
    }
}

// d_sca[c] = sum_p d_wt[p] |F(p, c)|^2 of the far fields d_F (far_field_launch's layout)
void sphere_sum_launch(const void* d_F, const double* d_wt, int npts, int nrhs, double* d_sca, cudaStream_t s) {
    k_sphere_sum<<<nrhs, 256, 0, s>>>((const double2*)d_F, d_wt, npts, d_sca);
    VIE_CHECK_LAUNCH();
}

void near_field_launch(Op& op, const void* d_I, int nrhs, const double* d_pts, int npts, void* d_out, cudaStream_t s) {
    const int groups = (nrhs + kRC - 1) / kRC;
    int pc = sum_cols(nrhs, npts);
    int nz = atom_chunks(op, (int64_t)pc * groups, 1);
    const int per = (op.N + nz - 1) / nz;
    nz = (op.N + per - 1) / per;
    pc = fit(op.d_fpart, (size_t)nz * nrhs * 3 * sizeof(double2), pc);
    for (int64_t p0 = 0; p0 < npts; p0 += pc) {
        const int P = (int)std::min<int64_t>(pc, npts - p0);
        k_near<<<dim3(P, nz, groups), 256, 0, s>>>(op.dmesh, geo_of(op), op.k, (const double2*)d_I, nrhs,
                                                   d_pts + 3 * p0, P, per, op.d_fpart.as<double2>());
        VIE_CHECK_LAUNCH();
        k_near_finish<<<(P * nrhs * 3 + 127) / 128, 128, 0, s>>>(op.d_fpart.as<double2>(), P, nrhs, nz, p0, npts,
                                                                 (double2*)d_out);
        VIE_CHECK_LAUNCH();
    }
}

}  // namespace vie
