// Three-dimensional operator build of the VIP method (the paper's introduction
// and Sec. 3: the method in three coordinates with the ten-term quadratic basis).
//
// Neighbour search (Sec. 3: nodes strictly inside |x_i - xbar| < rho), the MLS
// derivative weights of every node, VIP and normal point (Eq. fmlsrk:2 with the
// basis [1, xi, eta, zeta, xi^2, xi eta, xi zeta, eta^2, eta zeta, zeta^2]) and
// the operator tables of Eq. vip:1 and Sec. 4.1 (L, the six VIP interpolations,
// the VIP differences Gx, Gy, Gz, and the zero-normal-derivative rows of the
// boundary nodes).  Independent of the 2D context: its own handle (vip_3d),
// buffers and kernels.
//
// Layout: node coordinates, normals and spacing as FP64 structure-of-arrays.
// Points are enumerated as [nodes | 6 VIPs per interior node (E, W, N, S, T, B
// blocks of Ni each) | 2 normal points per boundary node (blocks of Nb)]; each
// point's neighbour list is a CSR row (int64 offsets, int32 node indices sorted
// ascending).  Node points carry 7 weight arrays (the derivative tables), the
// other points one (interpolation).  Tables are assembled as CSR on first use.
#include <cuda_pipeline.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <string>
#include <vector>

#include "vip_direct.cuh"
#include "../../include/vip.h"

struct vip_3d;

namespace {

constexpr int K3MAX = 160;                 // largest neighbour list per point
constexpr int NB3 = 10;                    // basis size
constexpr int NM3 = NB3 * (NB3 + 1) / 2;   // packed lower triangle of M
constexpr int NDER3 = 7;                   // node derivative tables
// Basis index of each node derivative table: (0,0,0) (1,0,0) (0,1,0) (0,0,1)
// (2,0,0) (0,2,0) (0,0,2) in the order of the basis above.
__constant__ int c_dbasis[NDER3] = {0, 1, 2, 3, 4, 7, 9};

struct Csr {
    int64_t* ptr = nullptr;
    int32_t* col = nullptr;
    double* val = nullptr;
    int64_t nnz = 0;
};

// Device view of the node set, the cell grid and the point enumeration.
struct Pts {
    const double *x, *y, *z, *nx, *ny, *nz, *h;
    const int32_t* interior;   // [Ni] node index of the k-th interior node
    const int32_t* boundary;   // [Nb] node index of the k-th boundary node
    int64_t N, Ni, Nb;
    double L[3];
    double support;
    int weight;
    double lo[3], cs[3];
    int nc[3];
    const int64_t* cell_ptr;   // [ncells + 1]
    const float4* cell_pts;    // [N] nodes sorted by cell: FP32 coordinates, node index (bits)
    float amax, Lf[3];         // bound of |coordinate| + L + rho; L (the FP32 test of distances)
};

__device__ __forceinline__ double min_img(double d, double L) {
    if (L <= 0.0) return d;
    double hl = 0.5 * L;
    if (d > hl) d = __dsub_rn(d, L);
    if (d < -hl) d = __dadd_rn(d, L);
    return d;
}

// Coordinates, dilation and owning node of point p (see the layout above).  The
// arithmetic is rounded step by step (no contraction), as the reference
// statement of the points is.
__device__ __forceinline__ void point_of(const Pts& a, int64_t p, double q[3], double& rho,
                                         int64_t& owner) {
    if (p < a.N) {
        owner = p;
        q[0] = a.x[p]; q[1] = a.y[p]; q[2] = a.z[p];
        rho = __dmul_rn(a.support, a.h[p]);
        return;
    }
    int64_t t = p - a.N;
    if (t < 6 * a.Ni) {
        int k = (int)(t / a.Ni);
        int64_t r = a.interior[t - (int64_t)k * a.Ni];
        owner = r;
        q[0] = a.x[r]; q[1] = a.y[r]; q[2] = a.z[r];
        double hh = __dmul_rn(0.5, a.h[r]);
        int ax = k >> 1;
        q[ax] = (k & 1) ? __dsub_rn(q[ax], hh) : __dadd_rn(q[ax], hh);
        rho = __dmul_rn(a.support, a.h[r]);
        return;
    }
    t -= 6 * a.Ni;
    int s = (int)(t / a.Nb);                   // 0: first normal point, 1: second
    int64_t r = a.boundary[t - (int64_t)s * a.Nb];
    owner = r;
    double sh = __dmul_rn((double)(s + 1), a.h[r]);
    q[0] = __dsub_rn(a.x[r], __dmul_rn(sh, a.nx[r]));
    q[1] = __dsub_rn(a.y[r], __dmul_rn(sh, a.ny[r]));
    q[2] = __dsub_rn(a.z[r], __dmul_rn(sh, a.nz[r]));
    rho = __dmul_rn(a.support, a.h[r]);
}

__device__ __forceinline__ int cell_coord(const Pts& a, double v, int ax) {
    double w;
    if (a.L[ax] > 0.0) w = v - floor(v / a.L[ax]) * a.L[ax];
    else w = v - a.lo[ax];
    int c = (int)floor(w / a.cs[ax]);
    return c < 0 ? 0 : (c >= a.nc[ax] ? a.nc[ax] - 1 : c);
}

// Is |x_j - q|^2 < rho^2 (minimum image in periodic sets)?  Decided in FP32 where that cannot
// be wrong, else by the FP64 test: the FP64 unit does two lanes a clock, and a point tests some
// 300 candidates (the FP64 tests alone took 3.9 ms of counting at 69,000 nodes).
// With u = 2^-24 and A bounding coordinates, L and rho, each FP32 offset is off by less than
// e = 16 u A, so squared distances near rho^2 by less than m = 8 (rho + e) e + 32 u rho^2; NaN
// and overflow fail both comparisons and are left to FP64.
struct PointSearch {       // what the search needs of a point, prepared once (k3_points)
    float q[3], in, out;   // FP32 coordinates; inside below `in`, outside above `out`
    int c[3];              // its cell
};

__global__ void k3_points(Pts a, int64_t P, PointSearch* __restrict__ out) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= P) return;
    double q[3], rho;
    int64_t owner;
    point_of(a, p, q, rho, owner);
    const float u = 5.9604645e-8f, rf = (float)rho;
    PointSearch t;
    float big = a.amax;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        t.q[k] = (float)q[k];
        big = fmaxf(big, fabsf(t.q[k]));
        t.c[k] = cell_coord(a, q[k], k);
    }
    const float e = 16.0f * u * big, r = rf * (1.0f + 4.0f * u);
    const float m = 8.0f * (r + e) * e + 32.0f * u * r * r;
    t.in = rf * rf - m;
    t.out = rf * rf + m;
    if (!(rf * rf > 1e-30f && rf * rf < 1e30f)) {  // squares out of FP32's normal range: all in FP64
        t.in = -1.0f;
        t.out = INFINITY;
    }
    out[p] = t;
}

__device__ __forceinline__ float image32(float d, float L) {
    if (L <= 0.0f) return d;
    if (d > 0.5f * L) d -= L;
    if (d < -0.5f * L) d += L;
    return d;
}
__device__ __noinline__ bool near64(const Pts& a, int64_t p, int nd) {
    double q[3], rho;
    int64_t owner;
    point_of(a, p, q, rho, owner);
    const double dx = min_img(__dsub_rn(a.x[nd], q[0]), a.L[0]);
    const double dy = min_img(__dsub_rn(a.y[nd], q[1]), a.L[1]);
    const double dz = min_img(__dsub_rn(a.z[nd], q[2]), a.L[2]);
    const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
    return d2 < __dmul_rn(rho, rho);
}
__device__ __forceinline__ bool near(const Pts& a, int64_t p, const PointSearch& t, const float4& c) {
    const float fx = image32(c.x - t.q[0], a.Lf[0]), fy = image32(c.y - t.q[1], a.Lf[1]),
                fz = image32(c.z - t.q[2], a.Lf[2]);
    const float f2 = fx * fx + fy * fy + fz * fz;
    if (f2 < t.in) return true;
    if (f2 > t.out) return false;
    return near64(a, p, __float_as_int(c.w));
}

__device__ __forceinline__ void flag(int* status, long long* bad, int code, int64_t p) {
    atomicCAS(status, 0, code);
    atomicMin(bad, (long long)p);
}

__global__ void k3_cell_count(Pts a, int64_t* __restrict__ node_cell, int32_t* __restrict__ cnt) {
    int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= a.N) return;
    int cx = cell_coord(a, a.x[r], 0), cy = cell_coord(a, a.y[r], 1), cz = cell_coord(a, a.z[r], 2);
    int64_t cell = ((int64_t)cx * a.nc[1] + cy) * a.nc[2] + cz;
    node_cell[r] = cell;
    atomicAdd(&cnt[cell], 1);
}

__global__ void k3_cell_fill(Pts a, const int64_t* __restrict__ node_cell, int32_t* __restrict__ cursor,
                             float4* __restrict__ cell_pts) {
    int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= a.N) return;
    int64_t c = node_cell[r];
    int pos = atomicAdd(&cursor[c], 1);
    cell_pts[a.cell_ptr[c] + pos] = make_float4((float)a.x[r], (float)a.y[r], (float)a.z[r], __int_as_float((int)r));
}

// Neighbours of point p, one warp per point: lanes 0 to 26 look up the cells around it, then
// the lanes test the candidates of all cells side by side.  Counting writes cnt[p]; filling
// gathers the list in shared memory and writes it in ascending node order (each lane counts the
// smaller entries).  Bound by the instructions of the candidate loop, about ten rounds a point.
// 459,000 points of 47 neighbours: count 0.46 ms, fill 0.65 ms (3.9 and 3.3 with a thread
// per point, FP64 tests and an insertion sort in global memory).
constexpr int NBR_WARPS = 4;
template <bool FILL>
__global__ void __launch_bounds__(32 * NBR_WARPS) k3_nbr(Pts a, int64_t P, int32_t* __restrict__ cnt, int* status,
                                                         long long* bad, const PointSearch* __restrict__ points,
                                                         const int64_t* __restrict__ pptr,
                                                         int32_t* __restrict__ pidx) {
    __shared__ int s_list[FILL ? NBR_WARPS : 1][FILL ? K3MAX : 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t p = (int64_t)blockIdx.x * NBR_WARPS + warp;
    if (p >= P) return;
    int64_t b = 0, e = 0;
    if (FILL) {
        b = pptr[p];
        e = pptr[p + 1];
        if (e == b) return;
    }
    const PointSearch pt = points[p];
    // lane l: cell (l / 9, l / 3 % 3, l % 3) of the neighbourhood
    int64_t cell = 0;
    bool have = lane < 27;
    const int off[3] = {lane / 9, lane / 3 % 3, lane % 3};
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        const int c = pt.c[ax], nc = a.nc[ax];
        int i;
        if (a.L[ax] > 0.0 && nc >= 3) {
            i = c - 1 + off[ax];
            i = i < 0 ? i + nc : i >= nc ? i - nc : i;
        } else if (a.L[ax] > 0.0) {
            i = off[ax];                       // every cell once
            have = have && i < nc;
        } else {
            i = c - 1 + off[ax];
            have = have && i >= 0 && i < nc;
        }
        cell = cell * nc + i;
    }
    const int64_t start = have ? a.cell_ptr[cell] : 0;
    const int len = have ? (int)(a.cell_ptr[cell + 1] - start) : 0;
    int end = len;                             // candidates of cells 0 .. lane
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, end, o);
        if (lane >= o) end += v;
    }
    const int total = __shfl_sync(0xffffffffu, end, 31);
    const int64_t shift = start - (end - len); // candidate m of this cell: cell_pts[shift + m]
    int n = 0;
    for (int m0 = 0; m0 < total; m0 += 32) {
        const int m = m0 + lane;
        int c = 0;                             // the first cell whose end lies beyond m
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const int v = __shfl_sync(0xffffffffu, end, c + o - 1);
            if (v <= m) c += o;
        }
        const int64_t at = __shfl_sync(0xffffffffu, shift, c) + m;
        bool in = false;
        int node = 0;
        if (m < total) {
            const float4 v = __ldg(a.cell_pts + at);
            node = __float_as_int(v.w);
            in = near(a, p, pt, v);
        }
        const unsigned hits = __ballot_sync(0xffffffffu, in);
        if (FILL && in) {
            const int k = n + __popc(hits & ((1u << lane) - 1u));
            if (k < K3MAX) s_list[warp][k] = node;
        }
        n += __popc(hits);
    }
    if (!FILL) {
        if (lane == 0) {
            if (n > K3MAX) {
                flag(status, bad, VIP_ERR_ARG, p);
                n = 0;
            }
            cnt[p] = n;
        }
        return;
    }
    __syncwarp();
    n = min(n, (int)(e - b));
    for (int k = lane; k < n; k += 32) {
        const int v = s_list[warp][k];
        int rank = 0;
        for (int j = 0; j < n; ++j) rank += s_list[warp][j] < v;
        pidx[b + rank] = v;
    }
}

// Weight at the scaled distance r >= 0.  The spline's two cubics are one Horner scheme with
// chosen coefficients; r is compared as an integer (doubles >= 0 order like their bits).
__device__ __forceinline__ double weight3(double r, int kind) {
    if (kind == VIP_W_PAPER) {
        if (r >= 1.0) return 0.0;
        double t = 1.0 - pow(r, (1.0 - r) * (1.0 - r));
        return (t * t) * (t * t);
    }
    const long long bits = __double_as_longlong(r);
    const bool inner = bits <= __double_as_longlong(0.5);
    const double c0 = inner ? 2.0 / 3.0 : 4.0 / 3.0, c1 = inner ? 0.0 : -4.0, c2 = inner ? -4.0 : 4.0,
                 c3 = inner ? 4.0 : -4.0 / 3.0;
    const double w = fma(r, fma(r, fma(r, c3, c2), c1), c0);
    return bits < __double_as_longlong(1.0) ? w : 0.0;
}

__device__ __forceinline__ constexpr int tri3(int i, int j) { return i * (i + 1) / 2 + j; }

// Basis vector at the scaled offset of neighbour node nd from point q (periodic: min_img).
__device__ __forceinline__ void basis_at(const Pts& a, int nd, const double q[3], double irho, bool periodic,
                                         double pv[NB3]) {
    double dx = a.x[nd] - q[0], dy = a.y[nd] - q[1], dz = a.z[nd] - q[2];
    if (periodic) {
        dx = min_img(dx, a.L[0]);
        dy = min_img(dy, a.L[1]);
        dz = min_img(dz, a.L[2]);
    }
    const double xi = dx * irho, eta = dy * irho, zeta = dz * irho;
    pv[0] = 1.0; pv[1] = xi; pv[2] = eta; pv[3] = zeta;
    pv[4] = xi * xi; pv[5] = xi * eta; pv[6] = xi * zeta;
    pv[7] = eta * eta; pv[8] = eta * zeta; pv[9] = zeta * zeta;
}

// Products p_i p_k of the basis are 35 monomials of degree <= 4, not 55: the place in the packed
// triangle of the first product equal to p_i p_k (i >= k).
__device__ __forceinline__ constexpr int same3(int i, int k) {
    switch (10 * i + k) {
        case 40: return tri3(1, 1);   // xx
        case 50: return tri3(2, 1);   // xy
        case 60: return tri3(3, 1);   // xz
        case 70: return tri3(2, 2);   // yy
        case 80: return tri3(3, 2);   // yz
        case 90: return tri3(3, 3);   // zz
        case 51: return tri3(4, 2);   // xxy
        case 61: return tri3(4, 3);   // xxz
        case 71: return tri3(5, 2);   // xyy
        case 62: case 81: return tri3(5, 3);   // xyz
        case 91: return tri3(6, 3);   // xzz
        case 82: return tri3(7, 3);   // yyz
        case 92: return tri3(8, 3);   // yzz
        case 74: return tri3(5, 5);   // xxyy
        case 84: return tri3(6, 5);   // xxyz
        case 94: return tri3(6, 6);   // xxzz
        case 85: return tri3(7, 6);   // xyyz
        case 95: return tri3(8, 6);   // xyzz
        case 97: return tri3(8, 8);   // yyzz
        default: return tri3(i, k);
    }
}

// MLS weights of every point: M = sum_j Phi_j p_j p_j^T (ten-term basis), its
// Cholesky factor, and for each derivative k wanted the vector z_k = M^{-1} e_k;
// then Psi_k(j) = fac_k Phi_j (z_k . p_j), fac_k = a! b! c! rho^-(a+b+c).
// Bound by the FP64 unit (two lanes a clock): so every sum of M is formed once, Phi_j is kept
// from the first pass over the neighbours in the place of the first weight, the nine z_k of a
// node share one pass, and divisions by rho and by the factor's diagonal are products with
// reciprocals.  69,000 nodes, 459,000 points: 4.4 ms (11.9 without).
__global__ void __launch_bounds__(128) k3_mls(Pts a, int64_t P, const int64_t* __restrict__ pptr,
                                              const int32_t* __restrict__ pidx,
                                              double* wnode, int64_t nnz_nodes,
                                              double* w0, int* status, long long* bad) {
    int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= P) return;
    int64_t b = pptr[p], e = pptr[p + 1];
    double q[3], rho;
    int64_t owner;
    point_of(a, p, q, rho, owner);
    const double irho = 1.0 / rho;
    const bool periodic = a.L[0] > 0.0 || a.L[1] > 0.0 || a.L[2] > 0.0;
    const bool node = p < a.N;
    double* wout = node ? wnode : w0 - nnz_nodes;
    double M[NM3];
#pragma unroll
    for (int i = 0; i < NM3; ++i) M[i] = 0.0;
    for (int64_t s = b; s < e; ++s) {
        double pv[NB3];
        basis_at(a, pidx[s], q, irho, periodic, pv);
        const double W = weight3(sqrt(pv[4] + pv[7] + pv[9]), a.weight);
        wout[s] = W;
#pragma unroll
        for (int i = 0; i < NB3; ++i) {
            double wi = W * pv[i];
#pragma unroll
            for (int k = 0; k <= i; ++k)
                if (same3(i, k) == tri3(i, k)) M[tri3(i, k)] = fma(wi, pv[k], M[tri3(i, k)]);
        }
    }
#pragma unroll
    for (int i = 0; i < NB3; ++i)
#pragma unroll
        for (int k = 0; k <= i; ++k) M[tri3(i, k)] = M[same3(i, k)];
    double trace = 0.0;
#pragma unroll
    for (int i = 0; i < NB3; ++i) trace += M[tri3(i, i)];
    bool ok = e > b;
#pragma unroll
    for (int j = 0; j < NB3; ++j) {
        double d = M[tri3(j, j)];
#pragma unroll
        for (int k = 0; k < j; ++k) d -= M[tri3(j, k)] * M[tri3(j, k)];
        if (!(d > 1e-13 * trace)) { ok = false; d = 1.0; }
        const double lj = sqrt(d), il = 1.0 / lj;
        M[tri3(j, j)] = il;                    // the reciprocal: all that the factor's diagonal is used for
#pragma unroll
        for (int i = j + 1; i < NB3; ++i) {
            double s = M[tri3(i, j)];
#pragma unroll
            for (int k = 0; k < j; ++k) s -= M[tri3(i, k)] * M[tri3(j, k)];
            M[tri3(i, j)] = s * il;
        }
    }
    if (!ok) {
        flag(status, bad, VIP_ERR_SINGULAR_STENCIL, p);
        return;
    }
    // fac_k z_k, z_k = M^{-1} e_k: L y = e_k, then L^T z = y
    double Z[NDER3][NB3];
    const int nk = node ? NDER3 : 1;
#pragma unroll 1
    for (int kk = 0; kk < nk; ++kk) {
        const int kb = c_dbasis[kk];
        double z[NB3];
#pragma unroll
        for (int i = 0; i < NB3; ++i) {
            double s = (i == kb) ? 1.0 : 0.0;
#pragma unroll
            for (int m = 0; m < i; ++m) s -= M[tri3(i, m)] * z[m];
            z[i] = s * M[tri3(i, i)];
        }
#pragma unroll
        for (int i = NB3 - 1; i >= 0; --i) {
            double s = z[i];
#pragma unroll
            for (int m = i + 1; m < NB3; ++m) s -= M[tri3(m, i)] * z[m];
            z[i] = s * M[tri3(i, i)];
        }
        const double fac = kb == 0 ? 1.0 : kb <= 3 ? irho : 2.0 * irho * irho;
#pragma unroll
        for (int i = 0; i < NB3; ++i) Z[kk][i] = fac * z[i];
    }
    if (!node) {
        double z[NB3];
#pragma unroll
        for (int i = 0; i < NB3; ++i) z[i] = Z[0][i];
        for (int64_t s = b; s < e; ++s) {
            double pv[NB3];
            basis_at(a, pidx[s], q, irho, periodic, pv);
            double dot = z[0];
#pragma unroll
            for (int i = 1; i < NB3; ++i) dot = fma(z[i], pv[i], dot);
            wout[s] *= dot;
        }
        return;
    }
    for (int64_t s = b; s < e; ++s) {
        double pv[NB3];
        basis_at(a, pidx[s], q, irho, periodic, pv);
        const double W = wout[s];
#pragma unroll
        for (int kk = 0; kk < NDER3; ++kk) {
            double dot = Z[kk][0];
#pragma unroll
            for (int i = 1; i < NB3; ++i) dot = fma(Z[kk][i], pv[i], dot);
            wnode[(int64_t)kk * nnz_nodes + s] = W * dot;
        }
    }
}

// ---- table assembly -------------------------------------------------------
struct Asm {
    Pts a;
    const int64_t* pptr;
    const int32_t* pidx;
    const double* wnode;
    const double* w0;
    int64_t nnz_nodes;
    const int32_t* ipos;   // [N] position in the interior list or -1
    const int32_t* bpos;   // [N] position in the boundary list or -1
};

// The two sorted source lists of row r for the merged tables: op GX/GY/GZ (the
// VIP pair of the axis) or NEUMANN (the two normal points).  Returns false for
// rows without entries.
__device__ __forceinline__ bool row_sources(const Asm& A, int op, int64_t r, int64_t& p1, int64_t& p2) {
    if (op == VIP3_OP_NEUMANN) {
        int32_t i = A.bpos[r];
        if (i < 0) return false;
        p1 = A.a.N + 6 * A.a.Ni + i;
        p2 = p1 + A.a.Nb;
        return true;
    }
    int32_t i = A.ipos[r];
    if (i < 0) return false;
    int ax = op - VIP3_OP_GX;
    p1 = A.a.N + (int64_t)(2 * ax) * A.a.Ni + i;
    p2 = p1 + A.a.Ni;
    return true;
}

// Walks the union of the two lists (and, for NEUMANN, the row's own node) in
// ascending column order, calling f(col, value).
template <class F>
__device__ __forceinline__ void merge_row(const Asm& A, int op, int64_t r, F f) {
    int64_t p1, p2;
    if (!row_sources(A, op, r, p1, p2)) return;
    int64_t i1 = A.pptr[p1], e1 = A.pptr[p1 + 1], i2 = A.pptr[p2], e2 = A.pptr[p2 + 1];
    const int64_t off = A.nnz_nodes;
    if (op == VIP3_OP_NEUMANN) {
        // q_r - (4/3) q(probe 1) + (1/3) q(probe 2), summed in that order
        bool diag = false;
        while (i1 < e1 || i2 < e2 || !diag) {
            int32_t c1 = i1 < e1 ? A.pidx[i1] : INT32_MAX;
            int32_t c2 = i2 < e2 ? A.pidx[i2] : INT32_MAX;
            int32_t cd = diag ? INT32_MAX : (int32_t)r;
            int32_t c = min(cd, min(c1, c2));
            double v = (c == cd) ? 1.0 : 0.0;
            if (c == cd) diag = true;
            if (c == c1) { v = __dsub_rn(v, __dmul_rn(4.0 / 3.0, A.w0[i1 - off])); ++i1; }
            else v = __dsub_rn(v, 0.0);
            if (c == c2) { v = __dadd_rn(v, __dmul_rn(1.0 / 3.0, A.w0[i2 - off])); ++i2; }
            f(c, v);
        }
        return;
    }
    const int ax = op - VIP3_OP_GX;
    double qa[3], qb[3], rho;
    int64_t owner;
    point_of(A.a, p1, qa, rho, owner);
    point_of(A.a, p2, qb, rho, owner);
    const double inv = 1.0 / fabs(__dsub_rn(qa[ax], qb[ax]));
    while (i1 < e1 || i2 < e2) {
        int32_t c1 = i1 < e1 ? A.pidx[i1] : INT32_MAX;
        int32_t c2 = i2 < e2 ? A.pidx[i2] : INT32_MAX;
        int32_t c = min(c1, c2);
        double v;
        if (c1 == c2) { v = __dsub_rn(A.w0[i1 - off], A.w0[i2 - off]); ++i1; ++i2; }
        else if (c == c1) { v = A.w0[i1 - off]; ++i1; }
        else { v = -A.w0[i2 - off]; ++i2; }
        f(c, __dmul_rn(v, inv));
    }
}

__global__ void k3_merge_count(Asm A, int op, int32_t* __restrict__ rowlen) {
    int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= A.a.N) return;
    int n = 0;
    merge_row(A, op, r, [&](int32_t, double) { ++n; });
    rowlen[r] = n;
}

__global__ void k3_merge_fill(Asm A, int op, const int64_t* __restrict__ ptr, int32_t* __restrict__ col,
                              double* __restrict__ val) {
    int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= A.a.N) return;
    int64_t w = ptr[r];
    const int64_t e = ptr[r + 1];
    merge_row(A, op, r, [&](int32_t c, double v) {
        if (w < e) { col[w] = c; val[w] = v; ++w; }
    });
}

// Rows of the VIP interpolation table k: the VIP's own list at interior rows.
__global__ void k3_vip_count(Asm A, int k, int32_t* __restrict__ rowlen) {
    int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= A.a.N) return;
    int32_t i = A.ipos[r];
    int n = 0;
    if (i >= 0) {
        int64_t p = A.a.N + (int64_t)k * A.a.Ni + i;
        n = (int)(A.pptr[p + 1] - A.pptr[p]);
    }
    rowlen[r] = n;
}

__global__ void k3_vip_fill(Asm A, int k, const int64_t* __restrict__ ptr, int32_t* __restrict__ col,
                            double* __restrict__ val) {
    int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= A.a.N) return;
    int32_t i = A.ipos[r];
    if (i < 0) return;
    int64_t p = A.a.N + (int64_t)k * A.a.Ni + i;
    int64_t w = ptr[r];
    for (int64_t s = A.pptr[p]; s < A.pptr[p + 1]; ++s, ++w) {
        col[w] = A.pidx[s];
        val[w] = A.w0[s - A.nnz_nodes];
    }
}

// Node tables: NBR (value 1), D000..D002, LAPLACE = (D200 + D020) + D002.
__global__ void k3_node_vals(Asm A, int op, double* __restrict__ val) {
    int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= A.nnz_nodes) return;
    double v;
    if (op == VIP3_OP_NBR) v = 1.0;
    else if (op == VIP3_OP_LAPLACE)
        v = __dadd_rn(__dadd_rn(A.wnode[4 * A.nnz_nodes + s], A.wnode[5 * A.nnz_nodes + s]),
                      A.wnode[6 * A.nnz_nodes + s]);
    else v = A.wnode[(int64_t)(op - VIP3_OP_D000) * A.nnz_nodes + s];
    val[s] = v;
}

__global__ void k3_csr_apply(int64_t n, const int64_t* __restrict__ ptr, const int32_t* __restrict__ col,
                             const double* __restrict__ val, const double* __restrict__ x,
                             double* __restrict__ y) {
    int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    double s = 0.0;
    for (int64_t k = ptr[r]; k < ptr[r + 1]; ++k) s = fma(val[k], x[col[k]], s);
    y[r] = s;
}

// ---- exclusive scan of int32 counts into int64 offsets (out[n] = total) ----
constexpr int SCAN_T = 256, SCAN_E = 4, SCAN_CHUNK = SCAN_T * SCAN_E;

__device__ __forceinline__ int64_t block_excl_scan(int64_t v, int64_t* sh, int64_t* total) {
    const int t = threadIdx.x;
    sh[t] = v;
    __syncthreads();
    for (int o = 1; o < SCAN_T; o <<= 1) {
        int64_t add = t >= o ? sh[t - o] : 0;
        __syncthreads();
        sh[t] += add;
        __syncthreads();
    }
    int64_t incl = sh[t];
    *total = sh[SCAN_T - 1];
    __syncthreads();
    return incl - v;
}

__global__ void __launch_bounds__(SCAN_T) k3_scan_local(const int32_t* __restrict__ in, int64_t n,
                                                        int64_t* __restrict__ out,
                                                        int64_t* __restrict__ bsum) {
    __shared__ int64_t sh[SCAN_T];
    const int64_t base = (int64_t)blockIdx.x * SCAN_CHUNK + (int64_t)threadIdx.x * SCAN_E;
    int64_t v[SCAN_E], s = 0;
#pragma unroll
    for (int k = 0; k < SCAN_E; ++k) {
        v[k] = base + k < n ? in[base + k] : 0;
        s += v[k];
    }
    int64_t tot;
    int64_t run = block_excl_scan(s, sh, &tot);
#pragma unroll
    for (int k = 0; k < SCAN_E; ++k) {
        if (base + k < n) out[base + k] = run;
        run += v[k];
    }
    if (threadIdx.x == 0) bsum[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(SCAN_T) k3_scan_blocks(int64_t* __restrict__ bsum, int64_t nb,
                                                         int64_t* __restrict__ total) {
    __shared__ int64_t sh[SCAN_T];
    int64_t carry = 0;
    for (int64_t c0 = 0; c0 < nb; c0 += SCAN_T) {
        int64_t i = c0 + threadIdx.x;
        int64_t v = i < nb ? bsum[i] : 0;
        int64_t tot;
        int64_t ex = block_excl_scan(v, sh, &tot);
        if (i < nb) bsum[i] = carry + ex;
        carry += tot;
    }
    if (threadIdx.x == 0) *total = carry;
}

__global__ void k3_scan_add(int64_t* __restrict__ out, int64_t n, const int64_t* __restrict__ boff) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] += boff[i / SCAN_CHUNK];
}

// ---- the fractional step in 3D (Sec. 2, Eqs. 12-15) ----------------------
// The step reads four tables in slices of 32 rows (SELL-32: entry k of the row at position q
// at base[q / 32] + 32 k + q % 32), made from the point lists on the first step: a thread
// per row then reads columns and values coalesced, where CSR rows of ~45 entries put the
// 32 lanes of a warp on 32 lines per entry.  Rows are summed in the same order with the
// same operations as from CSR, so the sums are the same bits.
//   0     the solves' system: L at interior rows, the Neumann rows at walls
//   1..3  Gx, Gy, Gz at interior rows
// Rows stand in an order of their own (perm): interior rows and wall rows in slices apart,
// the wall slices spread evenly among the others.  A Neumann row is about twice as long as
// an interior one, and in node order every lattice line ends in two, so that every slice
// would be as wide as its wall rows.  The first interior node k0 is at position 0, the
// border row N at position 1: N's row is k0's own equation, k0's row is empty.
// All four are laid out with one pass over the rows for the lengths, one scan and one
// allocation, straight from the point lists (first step with 32^3 and 64^3 nodes 0.7 and 3.4 ms,
// 8.1 KB of device memory a node; twelve tables copied from CSR took 3.3 and 10.9 ms, 15.6 KB).
constexpr int NTAB = 4;
struct Sell3 {
    const int64_t* base = nullptr;    // [slices + 1]
    const int32_t* len = nullptr;     // [positions] entries of each row
    const int32_t* col = nullptr;
    const double* val = nullptr;
};

// perm[q]: row at position q (-1: none).  Slice k holds walls where floor((k + 1) nw / nsl)
// exceeds floor(k nw / nsl), nw of the nsl slices being walls.
__global__ void k3_perm(int64_t N, int64_t Ni, int64_t Nb, int64_t nsl, int64_t nw,
                        const int32_t* __restrict__ interior, const int32_t* __restrict__ boundary,
                        int32_t* __restrict__ perm) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= 32 * nsl) return;
    const int64_t k = q >> 5, j = k * nw / nsl;
    int32_t r = -1;
    if ((k + 1) * nw / nsl > j) {
        const int64_t i = 32 * j + (q & 31);
        if (i < Nb) r = boundary[i];
    } else {
        const int64_t i = 32 * (k - j) + (q & 31);   // k0, N, the other interior nodes
        if (i == 1) r = (int32_t)N;
        else if (i <= Ni) r = interior[i == 0 ? 0 : i - 1];
    }
    perm[q] = r;
}

// Entries of row r of table t in column order, f(column, value).
template <class F>
__device__ __forceinline__ void step_row(const Asm& A, int t, int64_t r, F f) {
    if (t > 0) {
        merge_row(A, VIP3_OP_GX + t - 1, r, f);
    } else if (A.ipos[r] < 0) {
        merge_row(A, VIP3_OP_NEUMANN, r, f);
    } else {
        for (int64_t s = A.pptr[r]; s < A.pptr[r + 1]; ++s)
            f(A.pidx[s], __dadd_rn(__dadd_rn(A.wnode[4 * A.nnz_nodes + s], A.wnode[5 * A.nnz_nodes + s]),
                                   A.wnode[6 * A.nnz_nodes + s]));
    }
}
// row of a position as the tables hold it: N stands for k0's equation, k0 for no row
__device__ __forceinline__ int64_t row_at(const int32_t* __restrict__ perm, int64_t q, int64_t N, int64_t k0) {
    const int32_t r = perm[q];
    return r == N ? k0 : r == k0 ? -1 : r;
}

// Lengths of the rows of table blockIdx.y, and its slices' sizes in size[t nsl ..]; the system's
// interior slices once more in size[4 nsl ..] (0 for wall slices).
__global__ void __launch_bounds__(128) k3_step_size(Asm A, const int32_t* __restrict__ perm, int64_t k0, int64_t nsl,
                                                    int32_t* __restrict__ len, int32_t* __restrict__ size) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;  // whole warps: a slice each
    const int t = blockIdx.y;
    if (q >= 32 * nsl) return;
    const int64_t r = row_at(perm, q, A.a.N, k0);
    int n = 0;
    bool wall = false;
    if (r >= 0) {
        wall = A.ipos[r] < 0;
        if (t == 0 && !wall) n = (int)(A.pptr[r + 1] - A.pptr[r]);
        else step_row(A, t, r, [&](int32_t, double) { ++n; });
    }
    len[t * 32 * nsl + q] = n;
    const int w = __reduce_max_sync(0xffffffffu, n);
    wall = __any_sync(0xffffffffu, wall);
    if ((q & 31) == 0) {
        size[t * nsl + (q >> 5)] = w * 32;
        if (t == 0) size[NTAB * nsl + (q >> 5)] = wall ? 0 : w * 32;
    }
}

__global__ void __launch_bounds__(128) k3_step_fill(Asm A, const int32_t* __restrict__ perm, int64_t k0, int64_t nsl,
                                                    const int64_t* __restrict__ base, int32_t* __restrict__ scol,
                                                    double* __restrict__ sval) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int t = blockIdx.y;
    if (q >= 32 * nsl) return;
    const int64_t* bt = base + t * nsl + (q >> 5);
    int64_t o = bt[0] + (q & 31);
    const int64_t r = row_at(perm, q, A.a.N, k0);
    if (r >= 0)
        step_row(A, t, r, [&](int32_t c, double v) {
            scol[o] = c;
            sval[o] = v;
            o += 32;
        });
    for (; o < bt[1]; o += 32) {
        scol[o] = 0;
        sval[o] = 0.0;
    }
}

// most[0]: entries of the tables; most[1], most[2]: the most that a solve block's slices hold of
// the system, of its interior slices.
__global__ void __launch_bounds__(256) k3_step_most(int64_t nsl, int nb, const int64_t* __restrict__ base,
                                                    unsigned long long* __restrict__ most) {
    const int t = threadIdx.x;
    unsigned long long m[2] = {0, 0};
    for (int64_t k = t; k < nb; k += blockDim.x)
        for (int i = 0; i < 2; ++i) {
            const int64_t* bs = base + (i ? NTAB * nsl : 0);
            m[i] = max(m[i], (unsigned long long)(bs[nsl * (k + 1) / nb] - bs[nsl * k / nb]));
        }
    for (int i = 0; i < 2; ++i) atomicMax(most + 1 + i, m[i]);
    if (t == 0) most[0] = (unsigned long long)base[NTAB * nsl];
}

// sum_k a_rk x[f][col_rk] for NF fields through one row, in entry order, one chain per
// field.  The chain is serial and each batch of entries two dependent trips (indices,
// gathers), so both run ahead of it: while batch k is added, batch k + 1's values and
// gathers and batch k + 2's indices are on their way.
template <int NF>
__device__ __forceinline__ void row_sums(const int32_t* __restrict__ col, const double* __restrict__ val, int len,
                                         const double* const (&x)[NF], double (&out)[NF]) {
    constexpr int U = NF == 1 ? 8 : 4;
    int c0[U], c1[U];
    double a0[U], a1[U], g0[NF][U], g1[NF][U];
    auto index = [&](int (&c)[U], int k0) {
#pragma unroll
        for (int u = 0; u < U; ++u) c[u] = k0 + u < len ? col[32 * (k0 + u)] : 0;
    };
    auto fetch = [&](const int (&c)[U], double (&a)[U], double (&g)[NF][U], int k0) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool in = k0 + u < len;
            a[u] = in ? val[32 * (k0 + u)] : 0.0;
#pragma unroll
            for (int f = 0; f < NF; ++f) g[f][u] = in ? x[f][c[u]] : 0.0;
        }
    };
    auto add = [&](const double (&a)[U], const double (&g)[NF][U], int k0) {
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (k0 + u < len) {
#pragma unroll
                for (int f = 0; f < NF; ++f) out[f] = fma(a[u], g[f][u], out[f]);
            }
    };
#pragma unroll
    for (int f = 0; f < NF; ++f) out[f] = 0.0;
    index(c0, 0);
    index(c1, U);
    fetch(c0, a0, g0, 0);
#pragma unroll 1
    for (int k0 = 0; k0 < len; k0 += 2 * U) {
        fetch(c1, a1, g1, k0 + U);
        index(c0, k0 + 2 * U);
        add(a0, g0, k0);
        fetch(c0, a0, g0, k0 + 2 * U);
        index(c1, k0 + 3 * U);
        add(a1, g1, k0 + U);
    }
}
template <int NF>
__device__ __forceinline__ void sell_sums(const Sell3& t, int64_t r, const double* const (&x)[NF], double (&out)[NF]) {
    const int64_t o = t.base[r >> 5] + (r & 31);
    row_sums<NF>(t.col + o, t.val + o, t.len[r], x, out);
}

struct Fields3 { double* f[3]; };

// Convection at every node (Sec. 4.1 item 1 in three coordinates): the products
// of the six VIP interpolations of (u, v, w), differenced across each VIP pair
// and divided by the pair distance.
//
// A block takes 32 consecutive interior nodes, a warp for each axis.  The warp copies the 32
// lists of a VIP to shared memory, CONV_E entries of each at a time and the next ones beside
// the sums, 16 lanes along a list; there every lane walks its own list.  So the lists need no
// sliced copy (3.4 KB a node).
constexpr int CONV_E = 16, CONV_P = 33;   // entries of a list in a chunk; pitch of an entry's 32 lists
__global__ void __launch_bounds__(96) k3_conv(Asm A, Fields3 u, Fields3 out) {
    __shared__ double s_val[3][2][CONV_E * CONV_P];
    __shared__ int32_t s_col[3][2][CONV_E * CONV_P];
    __shared__ double s_x[3][3][32], s_inv[3][32];
    const int lane = threadIdx.x & 31, ax = threadIdx.x >> 5;
    const int64_t i0 = 32 * (int64_t)blockIdx.x, i = i0 + lane, Ni = A.a.Ni;
    const bool in = i < Ni;
    double v[2][3], q[2][3], rho;
    int64_t owner;
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        const int64_t p = A.a.N + (int64_t)(2 * ax + side) * Ni + i, b0 = A.pptr[p - lane];
        const int b = in ? (int)(A.pptr[p] - b0) : 0, len = in ? (int)(A.pptr[p + 1] - b0) - b : 0;
        const int32_t* col = A.pidx + b0;
        const double* val = A.w0 - A.nnz_nodes + b0;
        const int longest = __reduce_max_sync(0xffffffffu, len);
        auto copy = [&](int k0) {   // entries k0 .. k0 + 15 of every list
            const int e = lane & (CONV_E - 1), k = k0 + e, buf = (k0 / CONV_E) & 1;
#pragma unroll
            for (int j = 0; j < 32; j += 2) {
                const int l = j + (lane >> 4), at = __shfl_sync(0xffffffffu, b, l) + k;
                if (k < __shfl_sync(0xffffffffu, len, l)) {
                    __pipeline_memcpy_async(&s_col[ax][buf][e * CONV_P + l], col + at, 4);
                    __pipeline_memcpy_async(&s_val[ax][buf][e * CONV_P + l], val + at, 8);
                }
            }
            __pipeline_commit();
        };
        double sum[3] = {0.0, 0.0, 0.0};
        __syncwarp();
        copy(0);
#pragma unroll 1
        for (int k0 = 0; k0 < longest; k0 += CONV_E) {
            __syncwarp();           // the chunk before last has been read
            copy(k0 + CONV_E);
            __pipeline_wait_prior(1);
            __syncwarp();
            const int buf = (k0 / CONV_E) & 1;
            const int32_t* sc = s_col[ax][buf] + lane;
            const double* sv = s_val[ax][buf] + lane;
            constexpr int U = 8;
#pragma unroll
            for (int h = 0; h < CONV_E; h += U) {
                double g[3][U];
#pragma unroll
                for (int w = 0; w < U; ++w) {
                    const bool on = k0 + h + w < len;
                    const int c = on ? sc[(h + w) * CONV_P] : 0;
#pragma unroll
                    for (int f = 0; f < 3; ++f) g[f][w] = on ? u.f[f][c] : 0.0;
                }
#pragma unroll
                for (int w = 0; w < U; ++w)
                    if (k0 + h + w < len) {
                        const double a = sv[(h + w) * CONV_P];
#pragma unroll
                        for (int f = 0; f < 3; ++f) sum[f] = fma(a, g[f][w], sum[f]);
                    }
            }
        }
        __pipeline_wait_prior(0);
#pragma unroll
        for (int f = 0; f < 3; ++f) v[side][f] = sum[f];
        if (in) point_of(A.a, p, q[side], rho, owner);
    }
    if (in) {
        const double d = ax == 0 ? q[0][0] - q[1][0] : ax == 1 ? q[0][1] - q[1][1] : q[0][2] - q[1][2];
        const double wa = ax == 0 ? v[0][0] : ax == 1 ? v[0][1] : v[0][2],
                     wb = ax == 0 ? v[1][0] : ax == 1 ? v[1][1] : v[1][2];
        s_inv[ax][lane] = 1.0 / fabs(d);
#pragma unroll
        for (int c = 0; c < 3; ++c) s_x[ax][c][lane] = wa * v[0][c] - wb * v[1][c];
    }
    __syncthreads();
    if (!in) return;
    double f = 0.0;                                   // warp c: component c, axes in order
    for (int k = 0; k < 3; ++k) f += s_x[k][ax][lane] * s_inv[k][lane];
    out.f[ax][A.a.interior[i]] = f;
}

// Right-hand sides of Eq. (12) times dt of the three components at interior rows:
// (I + alpha L) u^n - dt (1.5 N^n - 0.5 N^{n-1} + G p^n); wall rows: the node's
// boundary value.  star gets the solves' initial guess u^n.
// Thread per position of the tables; the position of row N takes node k0 (see row_at).
struct Tabs3 {
    Sell3 sys, g[3];
    const int32_t* perm;
    int64_t n, N, k0;        // positions, nodes, first interior node
    const int32_t* ipos;
};
__global__ void __launch_bounds__(128) k3_rhs(Tabs3 T, double alpha, double dt, Fields3 bc, Fields3 u, Fields3 Ncur,
                                              Fields3 Nprev, const double* __restrict__ p, Fields3 rhs, Fields3 star) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= T.n) return;
    const int64_t r = row_at(T.perm, q, T.N, T.k0);
    if (r < 0) return;
    const bool inside = T.ipos[r] >= 0;
    double Lu[3] = {0.0, 0.0, 0.0};
    if (inside) {
        const double* const x[3] = {u.f[0], u.f[1], u.f[2]};
        sell_sums<3>(T.sys, q, x, Lu);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const double uc = u.f[c][r];
        star.f[c][r] = uc;
        if (!inside) {                                // wall: the boundary value
            rhs.f[c][r] = bc.f[c][r];
            continue;
        }
        double Gp[1];
        const double* const x[1] = {p};
        sell_sums<1>(T.g[c], q, x, Gp);
        const double nab = 1.5 * Ncur.f[c][r] - 0.5 * Nprev.f[c][r];
        rhs.f[c][r] = (uc + alpha * Lu[c]) - dt * (nab + Gp[0]);
    }
}

// Eq. (13) right-hand side, bordered: b_i = (Gx u* + Gy v* + Gz w*)_i / dt at
// interior rows, 0 at wall rows, then b_N = b_k0 and b_k0 = 0 (k0 the first
// interior node).
__global__ void __launch_bounds__(128) k3_div(Tabs3 T, double dt, Fields3 us, double* __restrict__ b) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= T.n) return;
    const int64_t r = row_at(T.perm, q, T.N, T.k0);
    if (r < 0) return;
    if (T.ipos[r] < 0) { b[r] = 0.0; return; }        // wall rows: zero normal derivative = 0
    double d[3][1];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const double* const x[1] = {us.f[c]};
        sell_sums<1>(T.g[c], q, x, d[c]);
    }
    const double v = (d[0][0] + d[1][0] + d[2][0]) / dt;
    if (r == T.k0) { b[T.N] = v; b[r] = 0.0; }
    else b[r] = v;
}

// Eqs. (14)-(15): u = u* - dt G phi at interior rows; p = p + phi - alpha L phi
// at every node (a wall row's L from the point lists: the system has its Neumann row).
__global__ void __launch_bounds__(128) k3_project(Tabs3 T, Asm A, double alpha, double dt, const double* __restrict__ phi,
                                                  Fields3 us, Fields3 u, double* __restrict__ p) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= T.n) return;
    const int64_t r = row_at(T.perm, q, T.N, T.k0);
    if (r < 0) return;
    const double* const x[1] = {phi};
    const bool inside = T.ipos[r] >= 0;               // walls keep their values
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        double g[1] = {0.0};
        if (inside) sell_sums<1>(T.g[c], q, x, g);
        u.f[c][r] = inside ? us.f[c][r] - dt * g[0] : us.f[c][r];
    }
    double l[1] = {0.0};
    if (inside) {
        sell_sums<1>(T.sys, q, x, l);
    } else {
        for (int64_t s = A.pptr[r]; s < A.pptr[r + 1]; ++s)
            l[0] = fma(__dadd_rn(__dadd_rn(A.wnode[4 * A.nnz_nodes + s], A.wnode[5 * A.nnz_nodes + s]),
                                 A.wnode[6 * A.nnz_nodes + s]),
                       phi[A.pidx[s]], l[0]);
    }
    p[r] = (p[r] + phi[r]) - alpha * l[0];
}

// ---- the step's linear solves ---------------------------------------------
// The two systems, applied matrix-free from their tables:
//   HELM: y = x - alpha L x at interior rows, y = x at wall rows      (n = N)
//   POIS: the bordered Poisson system (n = N + 1, x_N = mu): interior rows
//         y_i = (L x)_i + mu, wall rows y_i = (-6/h_i^2) (Nb x)_i, y_k0 =
//         (-6/h_k0^2) x_k0, y_N = (L x)_k0 + mu.
// Both read table 0; the Helmholtz system passes its wall rows over and takes k0's row from
// the position of row N, the next one.
// k3_bicgstab<NS> solves NS right-hand sides of one system in one cooperative launch:
// unpreconditioned FP64 BiCGSTAB (van der Vorst 1992) to ||b - A x|| <= rtol ||b|| with the
// oracle's rules: restart with r_hat = r when |r_hat . r| or |r_hat . v| falls below 1e-12
// of the product of norms, and confirm convergence on the true residual.  x holds the
// initial guess.
//
// A block owns a run of slices.  The vectors (and the table, if it fits) stay in its shared
// memory for the whole solve; p and s, which other blocks gather from, also go to global
// memory.  An iteration is five phases between grid barriers, bounded by the FP64 pipe (two
// lanes per clock and SM: 45 entries x 216 rows take 2.8 us per application at 32^3) and by
// the barriers and reductions (about 2 us each).  Before, it was 14 launches of a
// captured graph per iteration and a host read every few.  Step, before and now: 32^3 ABC
// flow 3.2 -> 1.1 ms, 31^3 lid-driven cube (320 iterations) 27.8 -> 7.9 ms, 64^3 ABC flow
// 17.7 -> 9.3 ms.  The three velocity components share the table's reads and the barriers.
enum { OPK_HELM = 0, OPK_POIS = 1 };
constexpr int NV3 = 7;  // r, rhat, p, v, s, t, x
// what a block keeps of each of its positions: the vectors, the boundary rows' scale and Pos3
template <int NS>
constexpr size_t pos_bytes() { return (NV3 * NS + 1) * sizeof(double) + 16; }
enum { ROW_IN = 0, ROW_WALL = 1, ROW_PIN = 2 };
struct Pos3 { int row, kind, len, at; };  // row (-1: none), its kind, its entries, the first one's offset
struct Out3 {
    int32_t it, status;
    double relres;
};
template <int NS>
struct Solve3 {
    int kind;
    int64_t n, N, k0, nsl;
    const int32_t* perm;     // [32 nsl] row of each position, -1: none
    double alpha, rtol;
    int32_t max_it;
    Sell3 t;
    const int64_t* copied;   // [nsl + 1] a slice's place among those that a block copies to shared memory
    const int32_t* ipos;
    const double* h;
    const double* rhs[NS];
    double* x[NS];
    double* gp[NS];          // p and s of every row
    double* gs[NS];
    double* work;            // pos_bytes per position, if a block's do not fit shared memory
    int vec_smem, mat_smem;  // what the block keeps in shared memory
    double* part;            // [2][3 NS][blocks]
    uint32_t* bar;
    int32_t* status;         // a failed solve stops those after it
    Out3* out;
};

__device__ __forceinline__ unsigned ld_acq3(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Grid barrier of a cooperative launch: block 0 adds 2^31 - (blocks - 1), the others 1, so the
// counter's top bit flips when the last block arrives; every wait ends after 2 s.
__device__ __noinline__ bool grid_sync3(uint32_t* bar, unsigned nb, int32_t* status) {
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        ok = 1;
        const unsigned add = blockIdx.x == 0 ? 0x80000000u - (nb - 1u) : 1u;
        unsigned old;
        asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], %2;" : "=r"(old) : "l"(bar), "r"(add) : "memory");
        uint64_t t0, t;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
        for (unsigned k = 1; ((ld_acq3(bar) ^ old) & 0x80000000u) == 0; ++k) {
            if ((k & 63u) == 0) {
                asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
                if (t - t0 > 2000000000ull || *(volatile int32_t*)status == VIP_ERR_TIMEOUT) {
                    atomicExch(status, VIP_ERR_TIMEOUT);
                    ok = 0;
                    break;
                }
            }
        }
    }
    __syncthreads();
    return ok != 0;
}

enum { S3_RESID = 0, S3_RUN = 1, S3_DONE = 2 };
struct Sys3 {
    double rho, rho_old, alpha, omega, beta, rhat_norm, tol, bnorm, relres;
    int it, restarts, state, status, xadd, zero;
};

template <int NS, int NT3>
__global__ void __launch_bounds__(NT3, 1) k3_bicgstab(Solve3<NS> a) {
    constexpr int NW3 = NT3 / 32;
    extern __shared__ __align__(16) double sm[];
    constexpr int Q = 3;  // dot products of a phase, at most
    __shared__ double red[Q * NS][NT3];
    __shared__ double tot[Q * NS];
    __shared__ Sys3 S[NS];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nb = (int)gridDim.x;
    if (*(volatile int32_t*)a.status != 0) return;  // written before this launch: the same for all blocks
    const int64_t s0 = a.nsl * blockIdx.x / nb, s1 = a.nsl * (blockIdx.x + 1) / nb;
    const int64_t pos0 = s0 * 32;
    const int pitch = (int)((s1 - s0) * 32);
    double* vec = a.vec_smem ? sm : a.work + pos0 * (pos_bytes<NS>() / 8);
    auto V = [&](int v, int q) -> double* { return vec + (int64_t)(v * NS + q) * pitch; };
    enum { VR, VH, VP, VV, VS, VT, VX };
    double* scale = vec + (int64_t)NV3 * NS * pitch;
    Pos3* pos = reinterpret_cast<Pos3*>(scale + pitch);
    const int64_t e0 = a.t.base[s0];
    const double* val = a.t.val + e0;
    const int32_t* col = a.t.col + e0;
    if (a.mat_smem) {
        const int ne = (int)(a.copied[s1] - a.copied[s0]);
        double* sv = sm + (a.vec_smem ? (int64_t)(pos_bytes<NS>() / 8) * pitch : 0);
        int32_t* sc = reinterpret_cast<int32_t*>(sv + ne);
        for (int64_t s = s0 + warp; s < s1; s += NW3) {
            const int o = (int)(a.copied[s] - a.copied[s0]), n = (int)(a.copied[s + 1] - a.copied[s]);
            const int64_t e = a.t.base[s] - e0;
            for (int k = lane; k < n; k += 32) {
                sv[o + k] = val[e + k];
                sc[o + k] = col[e + k];
            }
        }
        val = sv;
        col = sc;
    }
    for (int i = tid; i < pitch; i += NT3) {
        int r = __ldg(a.perm + pos0 + i);
        if (r >= a.n) r = -1;
        int kind = ROW_IN;
        double sc = 1.0;
        if (r >= 0 && r < a.N && a.ipos[r] < 0) kind = ROW_WALL;
        if (a.kind == OPK_POIS && r == a.k0) kind = ROW_PIN;
        if (a.kind == OPK_POIS && kind != ROW_IN) sc = -6.0 / (a.h[r] * a.h[r]);
        const bool none = r < 0 || (a.kind == OPK_HELM ? kind == ROW_WALL : kind == ROW_PIN);
        const int next = a.kind == OPK_HELM && r == a.k0 ? 1 : 0;
        const int64_t at = a.mat_smem ? a.copied[s0 + (i >> 5)] - a.copied[s0] : a.t.base[s0 + (i >> 5)] - e0;
        pos[i] = Pos3{r, kind, none ? 0 : a.t.len[pos0 + i + next], (int)at + (i & 31) + next};
        scale[i] = sc;
        if (r >= 0)
#pragma unroll
            for (int q = 0; q < NS; ++q) V(VX, q)[i] = a.x[q][r];
    }
    auto row_of = [&](int i) -> int { return pos[i].row; };
    if (tid < NS) S[tid] = Sys3{};  // state S3_RESID
    __syncthreads();
    // A applied to NS gathered vectors at position i
    auto apply = [&](int i, const Pos3& p, const double* const (&in)[NS], double (&y)[NS]) {
        row_sums<NS>(col + p.at, val + p.at, p.len, in, y);
#pragma unroll
        for (int q = 0; q < NS; ++q) {
            if (a.kind == OPK_HELM) y[q] = p.kind == ROW_WALL ? in[q][p.row] : in[q][p.row] - a.alpha * y[q];
            else if (p.kind == ROW_PIN) y[q] = scale[i] * in[q][p.row];
            else y[q] = p.kind == ROW_WALL ? scale[i] * y[q] : y[q] + in[q][a.N];
        }
    };
    // totals of nq quantities per system (index Q q + k): each thread's sums, 8 or 16 of them
    // per lane of one warp, a butterfly, then the blocks' partials in block order (two
    // alternating sets)
    int pset = 0;
    auto reduce = [&](const double (&d)[Q * NS], int nq) -> bool {
#pragma unroll
        for (int k = 0; k < Q * NS; ++k)
            if (k % Q < nq) red[k][tid] = d[k];
        __syncthreads();
        double* part = a.part + (int64_t)pset * Q * NS * nb;
        pset ^= 1;
#pragma unroll 1
        for (int j = warp; j < nq * NS; j += NW3) {
            const int k = j / nq * Q + j % nq;
            const double* p = red[k] + lane;
            double w = 0.0;
#pragma unroll
            for (int t = 0; t < NT3; t += 256)
                w += ((p[t] + p[t + 32]) + (p[t + 64] + p[t + 96])) + ((p[t + 128] + p[t + 160]) + (p[t + 192] + p[t + 224]));
            for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
            if (lane == 0) __stcg(part + (int64_t)k * nb + blockIdx.x, w);
        }
        if (!grid_sync3(a.bar, (unsigned)nb, a.status)) return false;
#pragma unroll 1
        for (int j = warp; j < nq * NS; j += NW3) {
            const int k = j / nq * Q + j % nq;
            double w = 0.0;
            for (int b = lane; b < nb; b += 5 * 32) {
                double g[5];
#pragma unroll
                for (int u = 0; u < 5; ++u) g[u] = b + 32 * u < nb ? __ldcg(part + (int64_t)k * nb + b + 32 * u) : 0.0;
                w += ((g[0] + g[1]) + (g[2] + g[3])) + g[4];
            }
            for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
            if (lane == 0) tot[k] = w;
        }
        __syncthreads();
        return true;
    };
    static_assert(NT3 % 256 == 0, "eight values per lane at a time");
    constexpr double BRK = 1e-12;
    // a system's next direction, after (r_hat . r, r . r)
    auto top = [&](Sys3& st, double rho, double rr) {
        if (st.it >= a.max_it || fabs(rho) <= BRK * st.rhat_norm * sqrt(rr)) {
            st.state = S3_RESID;
            return;
        }
        st.rho = rho;
        st.it += 1;
        st.beta = (rho / st.rho_old) * (st.alpha / st.omega);
    };
    bool first = true, alive = true;
    while (alive) {
        if (__syncthreads_or(tid < NS && S[tid].state == S3_RESID)) {
            if (!first) {  // the iterate to global memory, where its neighbours gather it
                for (int i = tid; i < pitch; i += NT3) {
                    const int r = row_of(i);
                    if (r < 0) continue;
#pragma unroll
                    for (int q = 0; q < NS; ++q)
                        if (S[q].state == S3_RESID) {
                            double xv = V(VX, q)[i];
                            if (S[q].xadd) V(VX, q)[i] = xv = xv + S[q].alpha * V(VP, q)[i];
                            a.x[q][r] = xv;
                        }
                }
                if (!grid_sync3(a.bar, (unsigned)nb, a.status)) return;
            }
            double d[Q * NS] = {};
            for (int i = tid; i < pitch; i += NT3) {
                const Pos3 ps = pos[i];
                const int r = ps.row;
                if (r < 0) continue;
                const double* in[NS];
                double y[NS];
#pragma unroll
                for (int q = 0; q < NS; ++q) in[q] = a.x[q];
                apply(i, ps, in, y);
#pragma unroll
                for (int q = 0; q < NS; ++q)
                    if (S[q].state == S3_RESID) {
                        const double b = a.rhs[q][r], res = b - y[q];
                        V(VR, q)[i] = res;
                        V(VH, q)[i] = res;
                        V(VP, q)[i] = 0.0;
                        V(VV, q)[i] = 0.0;
                        d[Q * q] = fma(res, res, d[Q * q]);
                        d[Q * q + 1] = fma(b, b, d[Q * q + 1]);
                    }
            }
            if (!reduce(d, 2)) return;
            if (tid < NS && S[tid].state == S3_RESID) {
                Sys3& st = S[tid];
                const double rr = tot[Q * tid];
                st.xadd = 0;
                if (first) {
                    st.bnorm = sqrt(tot[Q * tid + 1]);
                    st.tol = a.rtol * st.bnorm;
                }
                const double rn = sqrt(rr);
                if (!isfinite(st.bnorm)) {
                    st.state = S3_DONE;
                    st.status = VIP_ERR_NONFINITE;
                } else if (st.bnorm == 0.0) {  // x = 0 solves A x = 0
                    st.state = S3_DONE;
                    st.zero = 1;
                } else if (!isfinite(rr)) {
                    st.state = S3_DONE;
                    st.status = VIP_ERR_NONFINITE;
                } else if (rn <= st.tol || st.it >= a.max_it) {
                    st.state = S3_DONE;
                    st.relres = rn / st.bnorm;
                    if (rn > st.tol && st.relres > a.rtol) st.status = VIP_ERR_NOT_CONVERGED;
                } else if (++st.restarts > 1000) {
                    st.state = S3_DONE;
                    st.status = VIP_ERR_BREAKDOWN;
                } else {
                    st.state = S3_RUN;
                    st.rho_old = st.alpha = st.omega = 1.0;
                    st.rhat_norm = rn;
                    top(st, rr, rr);
                }
            }
            first = false;
            if (__syncthreads_or(tid < NS && S[tid].state == S3_RESID)) continue;
        }
        if (!__syncthreads_or(tid < NS && S[tid].state == S3_RUN)) break;
        // v = A p, p = r + beta (p - omega v) (half 0), or t = A s, s = r - alpha v (half 1),
        // with their dot products; s . s is tested with those of t (a converged s wastes
        // the last application, and every iteration saves a reduction)
#pragma unroll 1
        for (int half = 0; half < 2; ++half) {
            double d[Q * NS] = {};
            for (int i = tid; i < pitch; i += NT3) {
                const int r = row_of(i);
                if (r < 0) continue;
#pragma unroll
                for (int q = 0; q < NS; ++q)
                    if (S[q].state == S3_RUN) {
                        const double rv = V(VR, q)[i], vv = V(VV, q)[i];
                        if (!half) {
                            const double pv = rv + S[q].beta * (V(VP, q)[i] - S[q].omega * vv);
                            V(VP, q)[i] = pv;
                            a.gp[q][r] = pv;
                        } else {
                            const double sv = rv - S[q].alpha * vv;
                            V(VS, q)[i] = sv;
                            a.gs[q][r] = sv;
                        }
                    }
            }
            if (!grid_sync3(a.bar, (unsigned)nb, a.status)) return;
            for (int i = tid; i < pitch; i += NT3) {
                const Pos3 ps = pos[i];
                const int r = ps.row;
                if (r < 0) continue;
                const double* in[NS];
                double y[NS];
#pragma unroll
                for (int q = 0; q < NS; ++q) in[q] = half ? a.gs[q] : a.gp[q];
                apply(i, ps, in, y);
#pragma unroll
                for (int q = 0; q < NS; ++q)
                    if (S[q].state == S3_RUN) {
                        V(half ? VT : VV, q)[i] = y[q];
                        const double c = V(half ? VS : VH, q)[i];
                        d[Q * q] = fma(c, y[q], d[Q * q]);              // r_hat . v or s . t
                        d[Q * q + 1] = fma(y[q], y[q], d[Q * q + 1]);   // v . v or t . t
                        if (half) d[Q * q + 2] = fma(c, c, d[Q * q + 2]);
                    }
            }
            if (!reduce(d, 2 + half)) return;
            if (tid < NS && S[tid].state == S3_RUN) {
                Sys3& st = S[tid];
                const double cy = tot[Q * tid], yy = tot[Q * tid + 1];
                if (!isfinite(cy) || !isfinite(yy)) {
                    st.state = S3_DONE;
                    st.status = VIP_ERR_NONFINITE;
                } else if (!half) {
                    if (fabs(cy) <= BRK * st.rhat_norm * sqrt(yy)) st.state = S3_RESID;
                    else st.alpha = st.rho / cy;
                } else if (sqrt(tot[Q * tid + 2]) <= st.tol || yy == 0.0) {
                    st.xadd = 1;  // x += alpha p
                    st.state = S3_RESID;
                } else {
                    st.omega = cy / yy;
                }
            }
            __syncthreads();
        }
        // x += alpha p + omega s;  r = s - omega t
        double d[Q * NS] = {};
        for (int i = tid; i < pitch; i += NT3) {
            if (row_of(i) < 0) continue;
#pragma unroll
            for (int q = 0; q < NS; ++q)
                if (S[q].state == S3_RUN) {
                    const double sv = V(VS, q)[i];
                    V(VX, q)[i] = V(VX, q)[i] + S[q].alpha * V(VP, q)[i] + S[q].omega * sv;
                    const double rv = sv - S[q].omega * V(VT, q)[i];
                    V(VR, q)[i] = rv;
                    d[Q * q] = fma(V(VH, q)[i], rv, d[Q * q]);
                    d[Q * q + 1] = fma(rv, rv, d[Q * q + 1]);
                }
        }
        if (!reduce(d, 2)) return;
        if (tid < NS && S[tid].state == S3_RUN) {
            Sys3& st = S[tid];
            const double rho = tot[Q * tid], rr = tot[Q * tid + 1];
            if (!isfinite(rho) || !isfinite(rr)) {
                st.state = S3_DONE;
                st.status = VIP_ERR_NONFINITE;
            } else if (sqrt(rr) <= st.tol || st.omega == 0.0) {
                st.state = S3_RESID;
            } else {
                st.rho_old = st.rho;
                top(st, rho, rr);
            }
        }
        __syncthreads();
    }
    for (int i = tid; i < pitch; i += NT3)
#pragma unroll
        for (int q = 0; q < NS; ++q)
            if (S[q].zero && row_of(i) >= 0) a.x[q][row_of(i)] = 0.0;
    if (blockIdx.x == 0 && tid < NS) {
        a.out[tid] = Out3{S[tid].it, S[tid].status, S[tid].relres};
        if (S[tid].status) atomicCAS(a.status, 0, S[tid].status);
    }
}

inline unsigned blocks_for(int64_t n, int t) { return (unsigned)std::max<int64_t>(1, (n + t - 1) / t); }

}  // namespace

// ---------------------------------------------------------------------------
// Handle
// ---------------------------------------------------------------------------
struct vip_3d {
    int device = 0;
    int sms = 0, smem = 0;            // multiprocessors; dynamic shared memory of a solve block
    cudaStream_t stream = nullptr;
    std::string err;
    int weight = VIP_W_CUBIC_SPLINE;
    double support = 2.2;
    int64_t N = 0, Ni = 0, Nb = 0;
    double L[3] = {0, 0, 0};
    double lo[3] = {0, 0, 0}, hi[3] = {0, 0, 0}, hmax = 0.0, h0 = 0.0;
    std::vector<void*> node_bufs;     // freed on a new node set
    std::vector<void*> build_bufs;    // freed on a new build
    double *x = nullptr, *y = nullptr, *z = nullptr, *nx = nullptr, *ny = nullptr, *nz = nullptr,
           *h = nullptr;
    int32_t *interior = nullptr, *boundary = nullptr, *ipos = nullptr, *bpos = nullptr;
    bool built = false;
    Pts pts{};
    int64_t P = 0, nnz_all = 0, nnz_nodes = 0;
    int64_t* pptr = nullptr;
    int32_t* pidx = nullptr;
    double* wnode = nullptr;
    double* w0 = nullptr;
    Csr tab[VIP3_OP_COUNT];
    bool have[VIP3_OP_COUNT] = {};
    // the 3D step (vip_3d_set_flow, vip_3d_set_state, vip_3d_step)
    bool flow = false, state = false, have_prev = false;
    double Re = 0.0, dt = 0.0, rtol = 1e-8;
    int32_t max_iters = 20000;
    std::vector<void*> state_bufs;    // freed on a new node set
    double* vel[3] = {nullptr, nullptr, nullptr};
    double* star[3] = {nullptr, nullptr, nullptr};
    double* Ncur[3] = {nullptr, nullptr, nullptr};
    double* Nprev[3] = {nullptr, nullptr, nullptr};
    double* bc[3] = {nullptr, nullptr, nullptr};  // wall values (the state set last)
    double *p = nullptr, *phi = nullptr;          // phi: N + 1 (mu last)
    int64_t k0 = -1;                              // first interior node
    bool other_kinds = false;                     // SLIP or OUTLET nodes present
    double* rhs[3] = {nullptr, nullptr, nullptr}; // right-hand sides, N + 1 each (Poisson: the first)
    double* gather[2][3] = {};                    // p and s of the solves, N + 1 each
    double* work = nullptr;                       // Krylov vectors of blocks that exceed shared memory
    double* dpart = nullptr;                      // dot-product partials
    Out3* dout = nullptr;                         // [4] results of a step's solves
    uint32_t* dbar = nullptr;                     // [2] barrier word, status
    // the step's tables in slices, made on the first step after a build
    bool sliced = false;
    Sell3 tab3[NTAB];
    int32_t* perm = nullptr;                      // their row order
    const int64_t* inner = nullptr;               // [nsl + 1] entries of the system's interior slices before each
    int64_t nsl = 0;                              // its slices
    int64_t ent_helm = 0, ent_pois = 0;           // most entries of a solve block's slices
    int64_t steps = 0;
    int32_t last_helm = 0, last_poisson = 0;
    double last_poisson_res = 0.0;
};

namespace {

vip_status fail(vip_3d* b, vip_status st, const std::string& msg) {
    b->err = msg;
    return st;
}

#define V3_CUDA(call)                                                                      \
    do {                                                                                   \
        cudaError_t e_ = (call);                                                           \
        if (e_ != cudaSuccess) {                                                           \
            (void)cudaGetLastError();                                                      \
            return fail(b, e_ == cudaErrorMemoryAllocation ? VIP_ERR_OOM : VIP_ERR_CUDA,   \
                        std::string(#call) + ": " + cudaGetErrorString(e_));              \
        }                                                                                  \
    } while (0)

template <class T>
cudaError_t alloc(std::vector<void*>& owner, T** p, size_t n) {
    void* q = nullptr;
    cudaError_t e = cudaMalloc(&q, std::max<size_t>(n, 1) * sizeof(T));
    if (e == cudaSuccess) owner.push_back(q);
    *p = static_cast<T*>(q);
    return e;
}

void free_all(std::vector<void*>& v) {
    for (void* p : v) cudaFree(p);
    v.clear();
}

void reset_build(vip_3d* b) {
    free_all(b->build_bufs);
    b->built = b->sliced = false;
    b->work = nullptr;
    for (int i = 0; i < VIP3_OP_COUNT; ++i) { b->tab[i] = Csr{}; b->have[i] = false; }
    b->pptr = nullptr; b->pidx = nullptr; b->wnode = nullptr; b->w0 = nullptr;
    b->P = b->nnz_all = b->nnz_nodes = 0;
}

struct DeviceScope {
    int prev = -1;
    bool ok = false;
    explicit DeviceScope(int d) {
        if (cudaGetDevice(&prev) == cudaSuccess) ok = cudaSetDevice(d) == cudaSuccess;
    }
    ~DeviceScope() { if (prev >= 0) cudaSetDevice(prev); }
};

// out[0..n] = exclusive scan of in[0..n) (out[n] = total); bsum: scan_blocks(n) entries of scratch.
int64_t scan_blocks(int64_t n) { return std::max<int64_t>(1, (n + SCAN_CHUNK - 1) / SCAN_CHUNK); }
void enqueue_scan(vip_3d* b, const int32_t* in, int64_t n, int64_t* out, int64_t* bsum) {
    const int64_t nb = scan_blocks(n);
    k3_scan_local<<<(unsigned)nb, SCAN_T, 0, b->stream>>>(in, n, out, bsum);
    k3_scan_blocks<<<1, SCAN_T, 0, b->stream>>>(bsum, nb, out + n);
    k3_scan_add<<<blocks_for(n, 256), 256, 0, b->stream>>>(out, n, bsum);
}
// The same with scratch of its own; *total_host gets the total.
vip_status scan_counts(vip_3d* b, const int32_t* in, int64_t n, int64_t* out, int64_t* total_host) {
    std::vector<void*> tmp;
    int64_t* bsum = nullptr;
    cudaError_t e = alloc(tmp, &bsum, scan_blocks(n));
    if (e != cudaSuccess) { free_all(tmp); V3_CUDA(e); }
    enqueue_scan(b, in, n, out, bsum);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(total_host, out + n, sizeof(int64_t), cudaMemcpyDeviceToHost, b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    free_all(tmp);
    V3_CUDA(e);
    return VIP_OK;
}

Asm asm_view(const vip_3d* b) {
    Asm A;
    A.a = b->pts;
    A.pptr = b->pptr;
    A.pidx = b->pidx;
    A.wnode = b->wnode;
    A.w0 = b->w0;
    A.nnz_nodes = b->nnz_nodes;
    A.ipos = b->ipos;
    A.bpos = b->bpos;
    return A;
}

vip_status assemble(vip_3d* b, int op) {
    if (b->have[op]) return VIP_OK;
    const int64_t N = b->N;
    Asm A = asm_view(b);
    Csr T;
    if (op <= VIP3_OP_LAPLACE) {
        V3_CUDA(alloc(b->build_bufs, &T.ptr, N + 1));
        V3_CUDA(cudaMemcpyAsync(T.ptr, b->pptr, (N + 1) * sizeof(int64_t), cudaMemcpyDeviceToDevice, b->stream));
        T.col = b->pidx;          // the node points' lists come first
        T.nnz = b->nnz_nodes;
        V3_CUDA(alloc(b->build_bufs, &T.val, T.nnz));
        k3_node_vals<<<blocks_for(T.nnz, 256), 256, 0, b->stream>>>(A, op, T.val);
        V3_CUDA(cudaGetLastError());
    } else {
        std::vector<void*> tmp;
        int32_t* rowlen = nullptr;
        cudaError_t e = alloc(tmp, &rowlen, N);
        if (e != cudaSuccess) { free_all(tmp); V3_CUDA(e); }
        const bool vip = op <= VIP3_OP_VIP_B;
        if (vip) k3_vip_count<<<blocks_for(N, 256), 256, 0, b->stream>>>(A, op - VIP3_OP_VIP_E, rowlen);
        else k3_merge_count<<<blocks_for(N, 128), 128, 0, b->stream>>>(A, op, rowlen);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = alloc(b->build_bufs, &T.ptr, N + 1);
        if (e != cudaSuccess) { free_all(tmp); V3_CUDA(e); }
        vip_status st = scan_counts(b, rowlen, N, T.ptr, &T.nnz);
        free_all(tmp);
        if (st != VIP_OK) return st;
        V3_CUDA(alloc(b->build_bufs, &T.col, T.nnz));
        V3_CUDA(alloc(b->build_bufs, &T.val, T.nnz));
        if (vip) k3_vip_fill<<<blocks_for(N, 256), 256, 0, b->stream>>>(A, op - VIP3_OP_VIP_E, T.ptr, T.col, T.val);
        else k3_merge_fill<<<blocks_for(N, 128), 128, 0, b->stream>>>(A, op, T.ptr, T.col, T.val);
        V3_CUDA(cudaGetLastError());
    }
    V3_CUDA(cudaStreamSynchronize(b->stream));
    b->tab[op] = T;
    b->have[op] = true;
    return VIP_OK;
}

#define V3_TRY(call)                          \
    do {                                      \
        vip_status s_ = (call);               \
        if (s_ != VIP_OK) return s_;          \
    } while (0)

// blocks of a solve over n rows: one per SM, at least a slice each
int solve_blocks(const vip_3d* b) { return (int)std::max<int64_t>(1, std::min<int64_t>(b->sms, b->nsl)); }

// The step's tables (see Sell3).
vip_status slice_tables(vip_3d* b) {
    if (b->sliced) return VIP_OK;
    const Asm A = asm_view(b);
    cudaStream_t st = b->stream;
    const int64_t ni = (b->Ni + 1 + 31) / 32, nw = (b->Nb + 31) / 32, nsl = b->nsl = ni + nw, q = 32 * nsl;
    int32_t *rows = nullptr, *size = nullptr;
    int64_t* base = nullptr;
    V3_CUDA(alloc(b->build_bufs, &rows, (1 + NTAB) * q));                  // perm, lengths
    V3_CUDA(alloc(b->build_bufs, &base, (NTAB + 1) * nsl + 1 + 3));        // offsets, then k3_step_most's results
    int32_t *perm = rows, *len = rows + q;
    int64_t* most = base + (NTAB + 1) * nsl + 1;
    const int64_t nb = scan_blocks((NTAB + 1) * nsl);
    std::vector<void*> tmp;
    cudaError_t e = alloc(tmp, &size, (NTAB + 1) * nsl + 2 * (nb + 1));    // slice sizes, the scan's block sums
    if (e != cudaSuccess) { free_all(tmp); V3_CUDA(e); }
    const dim3 g((unsigned)blocks_for(q, 128), NTAB);
    k3_perm<<<blocks_for(q, 256), 256, 0, st>>>(b->N, b->Ni, b->Nb, nsl, nw, b->interior, b->boundary, perm);
    k3_step_size<<<g, 128, 0, st>>>(A, perm, b->k0, nsl, len, size);
    int64_t* bsum = reinterpret_cast<int64_t*>(size + ((NTAB + 1) * nsl + 1) / 2 * 2);
    enqueue_scan(b, size, (NTAB + 1) * nsl, base, bsum);
    e = cudaMemsetAsync(most, 0, 3 * sizeof(int64_t), st);
    k3_step_most<<<1, 256, 0, st>>>(nsl, solve_blocks(b), base, (unsigned long long*)most);
    int64_t h[3] = {0, 0, 0};
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(h, most, sizeof(h), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    free_all(tmp);
    V3_CUDA(e);
    double* val = nullptr;
    V3_CUDA(alloc(b->build_bufs, &val, h[0] + (h[0] + 1) / 2));            // values, columns
    int32_t* col = reinterpret_cast<int32_t*>(val + h[0]);
    k3_step_fill<<<g, 128, 0, st>>>(A, perm, b->k0, nsl, base, col, val);
    V3_CUDA(cudaGetLastError());
    for (int t = 0; t < NTAB; ++t) b->tab3[t] = Sell3{base + t * nsl, len + t * q, col, val};
    b->perm = perm;
    b->inner = base + NTAB * nsl;
    b->ent_pois = h[1];
    b->ent_helm = h[2];
    b->sliced = true;
    return VIP_OK;
}

// Enqueue the solve of NS right-hand sides; results in dout[slot ..).
template <int NS, int NT3>
vip_status solve_with(vip_3d* b, int kind, double* const* x, int slot) {
    const int nb = solve_blocks(b);
    Solve3<NS> a{};
    a.kind = kind;
    a.n = kind == OPK_HELM ? b->N : b->N + 1;
    a.nsl = b->nsl;
    a.perm = b->perm;
    a.N = b->N; a.k0 = b->k0;
    a.alpha = b->dt / (2.0 * b->Re);
    a.rtol = b->rtol;
    a.max_it = b->max_iters;
    a.t = b->tab3[0];
    a.copied = kind == OPK_HELM ? b->inner : b->tab3[0].base;
    a.ipos = b->ipos;
    a.h = b->h;
    for (int q = 0; q < NS; ++q) {
        a.rhs[q] = b->rhs[q];
        a.x[q] = x[q];
        a.gp[q] = b->gather[0][q];
        a.gs[q] = b->gather[1][q];
    }
    a.part = b->dpart;
    a.bar = b->dbar;
    a.status = reinterpret_cast<int32_t*>(b->dbar + 1);
    a.out = b->dout + slot;
    // shared memory: the vectors of the block's rows first, then its part of the table
    const size_t most = (size_t)b->smem;
    const size_t vb = pos_bytes<NS>() * ((b->nsl + nb - 1) / nb) * 32;
    const size_t mb = (size_t)(kind == OPK_HELM ? b->ent_helm : b->ent_pois) * 12;
    size_t dyn = 0;
    if (vb <= most) { a.vec_smem = 1; dyn = vb; }
    if (dyn + mb <= most) { a.mat_smem = 1; dyn += mb; }
    if (!a.vec_smem) {
        if (!b->work) V3_CUDA(alloc(b->build_bufs, &b->work, pos_bytes<3>() / 8 * 32 * b->nsl));
        a.work = b->work;
    }
    V3_CUDA(cudaMemsetAsync(b->dbar, 0, sizeof(uint32_t), b->stream));
    void* args[] = {&a};
    V3_CUDA(cudaLaunchCooperativeKernel((const void*)k3_bicgstab<NS, NT3>, dim3(nb), dim3(NT3), args, dyn, b->stream));
    return VIP_OK;
}

// 256 threads while a warp holds at most two slices (fewer to synchronise and reduce over);
// 512 beyond, where the table streams from L2 or memory and more warps keep more of it in
// flight (884,736 nodes: 60.6 -> 38.9 ms per step).
template <int NS>
vip_status solve(vip_3d* b, int kind, double* const* x, int slot) {
    return b->nsl <= (int64_t)16 * solve_blocks(b) ? solve_with<NS, 256>(b, kind, x, slot)
                                                   : solve_with<NS, 512>(b, kind, x, slot);
}

// One fractional step (Eqs. 12-15) on a built node set of interior and wall nodes.
vip_status step_once(vip_3d* b) {
    const int64_t N = b->N;
    const unsigned g = blocks_for(32 * b->nsl, 128);
    cudaStream_t st = b->stream;
    const double alpha = b->dt / (2.0 * b->Re), dt = b->dt;
    auto fields = [](double* const* f) { return Fields3{{f[0], f[1], f[2]}}; };
    const Asm A = asm_view(b);
    const Tabs3 T{b->tab3[0], {b->tab3[1], b->tab3[2], b->tab3[3]}, b->perm, 32 * b->nsl, N, b->k0, b->ipos};
    k3_conv<<<blocks_for(b->Ni, 32), 96, 0, st>>>(A, fields(b->vel), fields(b->Ncur));
    V3_CUDA(cudaGetLastError());
    if (!b->have_prev)
        for (int c = 0; c < 3; ++c)
            V3_CUDA(cudaMemcpyAsync(b->Nprev[c], b->Ncur[c], N * sizeof(double), cudaMemcpyDeviceToDevice, st));
    k3_rhs<<<g, 128, 0, st>>>(T, alpha, dt, fields(b->bc), fields(b->vel), fields(b->Ncur), fields(b->Nprev), b->p,
                              fields(b->rhs), fields(b->star));
    V3_CUDA(cudaGetLastError());
    V3_CUDA(cudaMemsetAsync(b->dbar, 0, 2 * sizeof(uint32_t), st));
    V3_TRY(solve<3>(b, OPK_HELM, b->star, 0));
    for (int c = 0; c < 3; ++c) std::swap(b->Ncur[c], b->Nprev[c]);
    b->have_prev = true;
    k3_div<<<g, 128, 0, st>>>(T, dt, fields(b->star), b->rhs[0]);
    V3_CUDA(cudaGetLastError());
    V3_TRY(solve<1>(b, OPK_POIS, &b->phi, 3));
    k3_project<<<g, 128, 0, st>>>(T, A, alpha, dt, b->phi, fields(b->star), fields(b->vel), b->p);
    V3_CUDA(cudaGetLastError());
    Out3 out[4] = {};
    uint32_t word[2] = {0, 0};
    V3_CUDA(cudaMemcpyAsync(out, b->dout, sizeof(out), cudaMemcpyDeviceToHost, st));
    V3_CUDA(cudaMemcpyAsync(word, b->dbar, sizeof(word), cudaMemcpyDeviceToHost, st));
    V3_CUDA(cudaStreamSynchronize(st));
    switch ((int32_t)word[1]) {
        case VIP_OK: break;
        case VIP_ERR_NONFINITE: return fail(b, VIP_ERR_NONFINITE, "non-finite right-hand side, residual or solution");
        case VIP_ERR_BREAKDOWN: return fail(b, VIP_ERR_BREAKDOWN, "BiCGSTAB: no progress after 1000 restarts");
        case VIP_ERR_NOT_CONVERGED: return fail(b, VIP_ERR_NOT_CONVERGED, "BiCGSTAB hit its iteration limit");
        default: return fail(b, (vip_status)word[1], "a solve's grid barrier timed out");
    }
    b->last_helm = out[0].it + out[1].it + out[2].it;
    b->last_poisson = out[3].it;
    b->last_poisson_res = out[3].relres;
    ++b->steps;
    return VIP_OK;
}

bool finite_all(const std::vector<double>& v) {
    for (double d : v) if (!std::isfinite(d)) return false;
    return true;
}

}  // namespace

// ---------------------------------------------------------------------------
// C ABI
// ---------------------------------------------------------------------------
extern "C" {

vip_status vip_3d_create(vip_3d** out, int device, void* cuda_stream) {
    if (!out) return VIP_ERR_ARG;
    *out = nullptr;
    int nd = 0;
    if (cudaGetDeviceCount(&nd) != cudaSuccess || device < 0 || device >= nd) {
        (void)cudaGetLastError();
        return VIP_ERR_ARG;
    }
    vip_3d* b = new (std::nothrow) vip_3d();
    if (!b) return VIP_ERR_OOM;
    b->device = device;
    b->stream = static_cast<cudaStream_t>(cuda_stream);
    // shared memory a block may have, less the solve kernel's own (its static arrays)
    int optin = 0;
    cudaFuncAttributes fa{};
    DeviceScope ds(device);
    if (!ds.ok || cudaDeviceGetAttribute(&b->sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device) != cudaSuccess ||
        cudaFuncGetAttributes(&fa, k3_bicgstab<3, 512>) != cudaSuccess) {
        (void)cudaGetLastError();
        delete b;
        return VIP_ERR_CUDA;
    }
    b->smem = std::max(0, optin - (int)fa.sharedSizeBytes - 1024);
    // One limit for every handle on the device: it belongs to the kernel, not to a launch, so a
    // solve that set it to its own need could lower it under another thread's launch.
    for (const void* k : {(const void*)k3_bicgstab<1, 256>, (const void*)k3_bicgstab<1, 512>,
                          (const void*)k3_bicgstab<3, 256>, (const void*)k3_bicgstab<3, 512>})
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, b->smem) != cudaSuccess) {
            (void)cudaGetLastError();
            delete b;
            return VIP_ERR_CUDA;
        }
    *out = b;
    return VIP_OK;
}

void vip_3d_destroy(vip_3d* b) {
    if (!b) return;
    DeviceScope ds(b->device);
    free_all(b->build_bufs);
    free_all(b->node_bufs);
    free_all(b->state_bufs);
    delete b;
}

const char* vip_3d_last_error(const vip_3d* b) { return b ? b->err.c_str() : "null handle"; }

vip_status vip_3d_set_mls(vip_3d* b, int weight, double support) {
    if (!b) return VIP_ERR_ARG;
    if (weight != VIP_W_CUBIC_SPLINE && weight != VIP_W_PAPER)
        return fail(b, VIP_ERR_ARG, "weight must be VIP_W_CUBIC_SPLINE or VIP_W_PAPER");
    if (!(support > 1.0) || !std::isfinite(support)) return fail(b, VIP_ERR_ARG, "support must be > 1");
    b->weight = weight;
    b->support = support;
    reset_build(b);
    return VIP_OK;
}

vip_status vip_3d_set_nodes(vip_3d* b, int64_t n, const double* x, const double* y, const double* z,
                            const uint8_t* kind, const double* nx, const double* ny, const double* nz,
                            const double* h, double Lx, double Ly, double Lz) {
    if (!b) return VIP_ERR_ARG;
    if (n < 1 || n >= INT32_MAX) return fail(b, VIP_ERR_ARG, "node count out of range");
    if (!x || !y || !z || !kind || !nx || !ny || !nz || !h) return fail(b, VIP_ERR_ARG, "null array");
    const double Ls[3] = {Lx, Ly, Lz};
    const int nper = (Lx > 0) + (Ly > 0) + (Lz > 0);
    for (double l : Ls)
        if (!std::isfinite(l) || l < 0.0) return fail(b, VIP_ERR_ARG, "periods must be finite and >= 0");
    if (nper != 0 && nper != 3) return fail(b, VIP_ERR_ARG, "periodic in every direction or in none");
    DeviceScope ds(b->device);
    if (!ds.ok) return fail(b, VIP_ERR_CUDA, "cudaSetDevice failed");
    // stage on the host (the inputs may be host or device memory) and check
    std::vector<double> hx(n), hy(n), hz(n), hnx(n), hny(n), hnz(n), hh(n);
    std::vector<uint8_t> hk(n);
    const double* src[7] = {x, y, z, nx, ny, nz, h};
    std::vector<double>* dst[7] = {&hx, &hy, &hz, &hnx, &hny, &hnz, &hh};
    for (int i = 0; i < 7; ++i) V3_CUDA(cudaMemcpy(dst[i]->data(), src[i], n * sizeof(double), cudaMemcpyDefault));
    V3_CUDA(cudaMemcpy(hk.data(), kind, n, cudaMemcpyDefault));
    for (int i = 0; i < 7; ++i)
        if (!finite_all(*dst[i])) return fail(b, VIP_ERR_ARG, "non-finite input");
    std::vector<int32_t> interior, boundary, ipos(n, -1), bpos(n, -1);
    double hmax = 0.0;
    double lo[3] = {hx[0], hy[0], hz[0]}, hi[3] = {hx[0], hy[0], hz[0]};
    for (int64_t i = 0; i < n; ++i) {
        if (!(hh[i] > 0.0)) return fail(b, VIP_ERR_ARG, "h must be > 0");
        if (hk[i] > VIP_NODE_OUTLET) return fail(b, VIP_ERR_ARG, "unknown node kind");
        if (hk[i] == VIP_NODE_INTERIOR) {
            ipos[i] = (int32_t)interior.size();
            interior.push_back((int32_t)i);
        } else {
            if (nper) return fail(b, VIP_ERR_ARG, "a periodic node set has interior nodes only");
            bpos[i] = (int32_t)boundary.size();
            boundary.push_back((int32_t)i);
        }
        hmax = std::max(hmax, hh[i]);
        const double c[3] = {hx[i], hy[i], hz[i]};
        for (int k = 0; k < 3; ++k) {
            if (nper && !(c[k] >= 0.0 && c[k] < Ls[k]))
                return fail(b, VIP_ERR_ARG, "periodic coordinates must lie in [0, L)");
            lo[k] = std::min(lo[k], c[k]);
            hi[k] = std::max(hi[k], c[k]);
        }
    }
    reset_build(b);
    free_all(b->node_bufs);
    free_all(b->state_bufs);
    for (int c = 0; c < 3; ++c) b->vel[c] = b->star[c] = b->Ncur[c] = b->Nprev[c] = b->bc[c] = nullptr;
    for (int c = 0; c < 3; ++c) b->rhs[c] = b->gather[0][c] = b->gather[1][c] = nullptr;
    b->p = b->phi = b->dpart = nullptr;
    b->dout = nullptr;
    b->dbar = nullptr;
    b->state = b->have_prev = false;
    b->steps = 0;
    b->N = 0;
    double** dptr[7] = {&b->x, &b->y, &b->z, &b->nx, &b->ny, &b->nz, &b->h};
    for (int i = 0; i < 7; ++i) {
        V3_CUDA(alloc(b->node_bufs, dptr[i], n));
        V3_CUDA(cudaMemcpy(*dptr[i], dst[i]->data(), n * sizeof(double), cudaMemcpyHostToDevice));
    }
    V3_CUDA(alloc(b->node_bufs, &b->interior, interior.size()));
    V3_CUDA(alloc(b->node_bufs, &b->boundary, boundary.size()));
    V3_CUDA(alloc(b->node_bufs, &b->ipos, n));
    V3_CUDA(alloc(b->node_bufs, &b->bpos, n));
    if (!interior.empty())
        V3_CUDA(cudaMemcpy(b->interior, interior.data(), interior.size() * 4, cudaMemcpyHostToDevice));
    if (!boundary.empty())
        V3_CUDA(cudaMemcpy(b->boundary, boundary.data(), boundary.size() * 4, cudaMemcpyHostToDevice));
    V3_CUDA(cudaMemcpy(b->ipos, ipos.data(), n * 4, cudaMemcpyHostToDevice));
    V3_CUDA(cudaMemcpy(b->bpos, bpos.data(), n * 4, cudaMemcpyHostToDevice));
    b->N = n;
    b->Ni = (int64_t)interior.size();
    b->Nb = (int64_t)boundary.size();
    for (int k = 0; k < 3; ++k) { b->L[k] = Ls[k]; b->lo[k] = lo[k]; b->hi[k] = hi[k]; }
    b->hmax = hmax;
    b->h0 = hh[0];
    b->k0 = interior.empty() ? -1 : interior[0];
    b->other_kinds = false;
    for (int64_t i = 0; i < n; ++i)
        if (hk[i] == VIP_NODE_SLIP || hk[i] == VIP_NODE_OUTLET) b->other_kinds = true;
    return VIP_OK;
}

vip_status vip_3d_build(vip_3d* b) {
    if (!b) return VIP_ERR_ARG;
    if (b->N < 1) return fail(b, VIP_ERR_ARG, "no node set");
    DeviceScope ds(b->device);
    if (!ds.ok) return fail(b, VIP_ERR_CUDA, "cudaSetDevice failed");
    reset_build(b);
    const int64_t N = b->N;
    const double rmax = b->support * b->hmax;
    // cell grid: cells of side >= the largest rho, at most about 8 N cells
    Pts& a = b->pts;
    a = Pts{};
    a.x = b->x; a.y = b->y; a.z = b->z; a.nx = b->nx; a.ny = b->ny; a.nz = b->nz; a.h = b->h;
    a.interior = b->interior; a.boundary = b->boundary;
    a.N = N; a.Ni = b->Ni; a.Nb = b->Nb;
    a.support = b->support; a.weight = b->weight;
    int64_t ncell = 1;
    for (int k = 0; k < 3; ++k) {
        a.L[k] = b->L[k];
        double ext = a.L[k] > 0.0 ? a.L[k] : b->hi[k] - b->lo[k];
        a.lo[k] = a.L[k] > 0.0 ? 0.0 : b->lo[k];
        a.nc[k] = (int)std::max(1.0, std::min(1.0e6, std::floor(ext / rmax)));
    }
    while ((ncell = (int64_t)a.nc[0] * a.nc[1] * a.nc[2]) > 8 * N + 4096) {
        for (int k = 0; k < 3; ++k)
            if (a.nc[k] > 3) a.nc[k] = std::max(3, (int)(a.nc[k] / 1.26));
    }
    for (int k = 0; k < 3; ++k) {
        double ext = a.L[k] > 0.0 ? a.L[k] : b->hi[k] - b->lo[k];
        a.cs[k] = ext > 0.0 ? ext / a.nc[k] : 1.0;
        if (ext > 0.0 && a.cs[k] < rmax) a.cs[k] = rmax;   // rounding guard
    }
    std::vector<void*> tmp;
    auto tmp_fail = [&](cudaError_t e) { free_all(tmp); return e; };
    int64_t* node_cell = nullptr;
    int32_t *cnt = nullptr, *cursor = nullptr;
    int64_t* cell_ptr = nullptr;
    float4* cell_pts = nullptr;
    int* status = nullptr;
    long long* bad = nullptr;
    cudaError_t e = alloc(tmp, &node_cell, N);
    if (e == cudaSuccess) e = alloc(tmp, &cnt, ncell);
    if (e == cudaSuccess) e = alloc(tmp, &cursor, ncell);
    if (e == cudaSuccess) e = alloc(b->build_bufs, &cell_ptr, ncell + 1);
    if (e == cudaSuccess) e = alloc(b->build_bufs, &cell_pts, N);
    if (e == cudaSuccess) e = alloc(tmp, &status, 1);
    if (e == cudaSuccess) e = alloc(tmp, &bad, 1);
    if (e == cudaSuccess) e = cudaMemsetAsync(cnt, 0, ncell * sizeof(int32_t), b->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(cursor, 0, ncell * sizeof(int32_t), b->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(status, 0, sizeof(int), b->stream);
    const long long big = INT64_MAX;
    if (e == cudaSuccess) e = cudaMemcpyAsync(bad, &big, sizeof(long long), cudaMemcpyHostToDevice, b->stream);
    if (e != cudaSuccess) V3_CUDA(tmp_fail(e));
    a.cell_ptr = cell_ptr;
    a.cell_pts = cell_pts;
    double amax = rmax;
    for (int k = 0; k < 3; ++k)
        amax = std::max(amax, rmax + std::max({std::fabs(b->lo[k]), std::fabs(b->hi[k]), b->L[k]}) + b->L[k]);
    a.amax = (float)(amax * 1.000001);
    for (int k = 0; k < 3; ++k) a.Lf[k] = (float)a.L[k];
    k3_cell_count<<<blocks_for(N, 256), 256, 0, b->stream>>>(a, node_cell, cnt);
    if ((e = cudaGetLastError()) != cudaSuccess) V3_CUDA(tmp_fail(e));
    int64_t tot = 0;
    vip_status st = scan_counts(b, cnt, ncell, cell_ptr, &tot);
    if (st != VIP_OK) { free_all(tmp); return st; }
    k3_cell_fill<<<blocks_for(N, 256), 256, 0, b->stream>>>(a, node_cell, cursor, cell_pts);
    if ((e = cudaGetLastError()) != cudaSuccess) V3_CUDA(tmp_fail(e));
    // points and their neighbour lists
    const int64_t P = N + 6 * b->Ni + 2 * b->Nb;
    int32_t* pcnt = nullptr;
    if ((e = alloc(tmp, &pcnt, P)) != cudaSuccess) V3_CUDA(tmp_fail(e));
    if ((e = alloc(b->build_bufs, &b->pptr, P + 1)) != cudaSuccess) V3_CUDA(tmp_fail(e));
    PointSearch* points = nullptr;
    if ((e = alloc(tmp, &points, P)) != cudaSuccess) V3_CUDA(tmp_fail(e));
    k3_points<<<blocks_for(P, 128), 128, 0, b->stream>>>(a, P, points);
    k3_nbr<false><<<blocks_for(P, NBR_WARPS), 32 * NBR_WARPS, 0, b->stream>>>(a, P, pcnt, status, bad, points,
                                                                             nullptr, nullptr);
    if ((e = cudaGetLastError()) != cudaSuccess) V3_CUDA(tmp_fail(e));
    int hst = 0;
    long long hbad = 0;
    if ((e = cudaMemcpyAsync(&hst, status, sizeof(int), cudaMemcpyDeviceToHost, b->stream)) != cudaSuccess ||
        (e = cudaMemcpyAsync(&hbad, bad, sizeof(long long), cudaMemcpyDeviceToHost, b->stream)) != cudaSuccess ||
        (e = cudaStreamSynchronize(b->stream)) != cudaSuccess)
        V3_CUDA(tmp_fail(e));
    if (hst != 0) {
        free_all(tmp);
        return fail(b, (vip_status)hst, "point " + std::to_string(hbad) + " has more than " +
                                             std::to_string(K3MAX) + " neighbours");
    }
    int64_t nnz = 0;
    st = scan_counts(b, pcnt, P, b->pptr, &nnz);
    if (st != VIP_OK) { free_all(tmp); return st; }
    int64_t nnz_nodes = 0;
    if ((e = cudaMemcpy(&nnz_nodes, b->pptr + N, sizeof(int64_t), cudaMemcpyDeviceToHost)) != cudaSuccess)
        V3_CUDA(tmp_fail(e));
    if ((e = alloc(b->build_bufs, &b->pidx, nnz)) != cudaSuccess) V3_CUDA(tmp_fail(e));
    if ((e = alloc(b->build_bufs, &b->wnode, (size_t)NDER3 * nnz_nodes)) != cudaSuccess) V3_CUDA(tmp_fail(e));
    if ((e = alloc(b->build_bufs, &b->w0, nnz - nnz_nodes)) != cudaSuccess) V3_CUDA(tmp_fail(e));
    k3_nbr<true><<<blocks_for(P, NBR_WARPS), 32 * NBR_WARPS, 0, b->stream>>>(a, P, nullptr, status, bad, points,
                                                                            b->pptr, b->pidx);
    k3_mls<<<blocks_for(P, 128), 128, 0, b->stream>>>(a, P, b->pptr, b->pidx, b->wnode, nnz_nodes, b->w0,
                                                      status, bad);
    if ((e = cudaGetLastError()) != cudaSuccess) V3_CUDA(tmp_fail(e));
    if ((e = cudaMemcpyAsync(&hst, status, sizeof(int), cudaMemcpyDeviceToHost, b->stream)) != cudaSuccess ||
        (e = cudaMemcpyAsync(&hbad, bad, sizeof(long long), cudaMemcpyDeviceToHost, b->stream)) != cudaSuccess ||
        (e = cudaStreamSynchronize(b->stream)) != cudaSuccess)
        V3_CUDA(tmp_fail(e));
    free_all(tmp);
    if (hst != 0) return fail(b, (vip_status)hst, "moment matrix of point " + std::to_string(hbad) +
                                                      " failed its Cholesky test");
    b->P = P;
    b->nnz_all = nnz;
    b->nnz_nodes = nnz_nodes;
    b->built = true;
    return VIP_OK;
}

vip_status vip_3d_stencil_size(vip_3d* b, int which, int64_t* nrows, int64_t* nnz) {
    if (!b) return VIP_ERR_ARG;
    if (!b->built) return fail(b, VIP_ERR_ARG, "not built");
    if (which < 0 || which >= VIP3_OP_COUNT) return fail(b, VIP_ERR_ARG, "bad table");
    DeviceScope ds(b->device);
    vip_status st = assemble(b, which);
    if (st != VIP_OK) return st;
    if (nrows) *nrows = b->N;
    if (nnz) *nnz = b->tab[which].nnz;
    return VIP_OK;
}

vip_status vip_3d_get_stencil(vip_3d* b, int which, int64_t* row_ptr, int32_t* col, double* val) {
    vip_status st = vip_3d_stencil_size(b, which, nullptr, nullptr);
    if (st != VIP_OK) return st;
    if (!row_ptr || !col || !val) return fail(b, VIP_ERR_ARG, "null array");
    DeviceScope ds(b->device);
    const Csr& T = b->tab[which];
    V3_CUDA(cudaMemcpyAsync(row_ptr, T.ptr, (b->N + 1) * sizeof(int64_t), cudaMemcpyDefault, b->stream));
    if (T.nnz) {
        V3_CUDA(cudaMemcpyAsync(col, T.col, T.nnz * sizeof(int32_t), cudaMemcpyDefault, b->stream));
        V3_CUDA(cudaMemcpyAsync(val, T.val, T.nnz * sizeof(double), cudaMemcpyDefault, b->stream));
    }
    V3_CUDA(cudaStreamSynchronize(b->stream));
    return VIP_OK;
}

vip_status vip_3d_apply(vip_3d* b, int which, const double* x, double* y) {
    vip_status st = vip_3d_stencil_size(b, which, nullptr, nullptr);
    if (st != VIP_OK) return st;
    if (!x || !y) return fail(b, VIP_ERR_ARG, "null array");
    DeviceScope ds(b->device);
    const int64_t N = b->N;
    std::vector<void*> tmp;
    const Csr& T = b->tab[which];
    if (vip::direct_vectors(b->device, x, y, N)) {
        k3_csr_apply<<<blocks_for(N, 256), 256, 0, b->stream>>>(N, T.ptr, T.col, T.val, x, y);
        V3_CUDA(cudaGetLastError());
        V3_CUDA(cudaStreamSynchronize(b->stream));
        return VIP_OK;
    }
    double *dx = nullptr, *dy = nullptr;
    cudaError_t e = alloc(tmp, &dx, N);
    if (e == cudaSuccess) e = alloc(tmp, &dy, N);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dx, x, N * sizeof(double), cudaMemcpyDefault, b->stream);
    if (e == cudaSuccess) {
        k3_csr_apply<<<blocks_for(N, 256), 256, 0, b->stream>>>(N, T.ptr, T.col, T.val, dx, dy);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(y, dy, N * sizeof(double), cudaMemcpyDefault, b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    free_all(tmp);
    V3_CUDA(e);
    return VIP_OK;
}

vip_status vip_3d_set_flow(vip_3d* b, double Re, double dt, double rtol, int32_t max_iters) {
    if (!b) return VIP_ERR_ARG;
    if (!(Re > 0.0) || !(dt > 0.0) || !std::isfinite(Re) || !std::isfinite(dt))
        return fail(b, VIP_ERR_ARG, "Re and dt must be finite and > 0");
    if (!(rtol > 0.0 && rtol < 1.0)) return fail(b, VIP_ERR_ARG, "rtol must lie in (0, 1)");
    if (max_iters < 1) return fail(b, VIP_ERR_ARG, "max_iters must be >= 1");
    b->Re = Re;
    b->dt = dt;
    b->rtol = rtol;
    b->max_iters = max_iters;
    b->flow = true;
    return VIP_OK;
}

vip_status vip_3d_set_state(vip_3d* b, const double* u, const double* v, const double* w, const double* p) {
    if (!b) return VIP_ERR_ARG;
    if (b->N < 1) return fail(b, VIP_ERR_ARG, "no node set");
    if (!u || !v || !w || !p) return fail(b, VIP_ERR_ARG, "null array");
    DeviceScope ds(b->device);
    const int64_t N = b->N;
    if (!b->p) {
        for (int c = 0; c < 3; ++c) {
            V3_CUDA(alloc(b->state_bufs, &b->vel[c], N));
            V3_CUDA(alloc(b->state_bufs, &b->star[c], N));
            V3_CUDA(alloc(b->state_bufs, &b->Ncur[c], N));
            V3_CUDA(alloc(b->state_bufs, &b->Nprev[c], N));
            V3_CUDA(alloc(b->state_bufs, &b->bc[c], N));
        }
        V3_CUDA(alloc(b->state_bufs, &b->p, N));
        V3_CUDA(alloc(b->state_bufs, &b->phi, N + 1));
        for (int c = 0; c < 3; ++c) {
            V3_CUDA(alloc(b->state_bufs, &b->rhs[c], N + 1));
            V3_CUDA(alloc(b->state_bufs, &b->gather[0][c], N + 1));
            V3_CUDA(alloc(b->state_bufs, &b->gather[1][c], N + 1));
        }
        V3_CUDA(alloc(b->state_bufs, &b->dpart, (size_t)2 * 9 * b->sms));
        V3_CUDA(alloc(b->state_bufs, &b->dout, 4));
        V3_CUDA(alloc(b->state_bufs, &b->dbar, 2));
    }
    const double* src[4] = {u, v, w, p};
    double* dst[4] = {b->vel[0], b->vel[1], b->vel[2], b->p};
    for (int k = 0; k < 4; ++k)
        V3_CUDA(cudaMemcpyAsync(dst[k], src[k], N * sizeof(double), cudaMemcpyDefault, b->stream));
    for (int c = 0; c < 3; ++c)
        V3_CUDA(cudaMemcpyAsync(b->bc[c], b->vel[c], N * sizeof(double), cudaMemcpyDeviceToDevice, b->stream));
    V3_CUDA(cudaMemsetAsync(b->phi, 0, (N + 1) * sizeof(double), b->stream));
    V3_CUDA(cudaStreamSynchronize(b->stream));
    b->have_prev = false;
    b->state = true;
    b->steps = 0;
    return VIP_OK;
}

vip_status vip_3d_step(vip_3d* b, int32_t nsteps) {
    if (!b) return VIP_ERR_ARG;
    if (!b->built) return fail(b, VIP_ERR_ARG, "not built");
    if (!b->flow || !b->state) return fail(b, VIP_ERR_ARG, "vip_3d_set_flow and vip_3d_set_state first");
    if (b->other_kinds) return fail(b, VIP_ERR_ARG, "the 3D step takes interior and wall nodes only");
    if (b->k0 < 0) return fail(b, VIP_ERR_ARG, "the 3D step needs an interior node");
    if (nsteps < 0) return fail(b, VIP_ERR_ARG, "nsteps must be >= 0");
    DeviceScope ds(b->device);
    V3_TRY(slice_tables(b));
    for (int k = 0; k < nsteps; ++k) V3_TRY(step_once(b));
    return VIP_OK;
}

vip_status vip_3d_get_state(vip_3d* b, double* u, double* v, double* w, double* p, double* phi) {
    if (!b) return VIP_ERR_ARG;
    if (!b->state) return fail(b, VIP_ERR_ARG, "no state");
    DeviceScope ds(b->device);
    const int64_t N = b->N;
    double* dst[5] = {u, v, w, p, phi};
    const double* src[5] = {b->vel[0], b->vel[1], b->vel[2], b->p, b->phi};
    for (int k = 0; k < 5; ++k)
        if (dst[k]) V3_CUDA(cudaMemcpyAsync(dst[k], src[k], N * sizeof(double), cudaMemcpyDefault, b->stream));
    V3_CUDA(cudaStreamSynchronize(b->stream));
    return VIP_OK;
}

vip_status vip_3d_get_iters(vip_3d* b, int64_t* steps, int32_t* helm_iters, int32_t* poisson_iters,
                            double* poisson_relres) {
    if (!b) return VIP_ERR_ARG;
    if (steps) *steps = b->steps;
    if (helm_iters) *helm_iters = b->last_helm;
    if (poisson_iters) *poisson_iters = b->last_poisson;
    if (poisson_relres) *poisson_relres = b->last_poisson_res;
    return VIP_OK;
}

}  // extern "C"
