// Space-time HDG assembly on the GPU: element matrices of the bilinear form
// (arXiv:2010.11130, Section 2.3, eqs. st-hdg and bilin, upwind flux sigma_a
// and interior-penalty flux sigma_d of eq. IPpenalty), static condensation
// S_K = D_K - C_K A_K^{-1} B_K, H_K = G_K - C_K A_K^{-1} F_K (Section 2.5,
// eqs. linsys and systemLambda), scatter into the facet CSR pattern and the
// left scaling by the facet block-diagonal inverse (Section 4 settings).
//
// For an element K with test (v, mu) and trial (u, lambda), unit space-time
// normal n_hat = (n_t, n), a_hat = (1, a), a_hat_n = a_hat . n_hat,
// c+ = (a_hat_n + |a_hat_n|)/2, c- = (a_hat_n - |a_hat_n|)/2, pen = nu alpha / h_K
// (h_K the longest edge), the local blocks are
//   A(v, u)   = int_K -u a_hat.grad_hat v + nu grad u . grad v
//             + int_dK (c+ + pen) u v - nu (grad u . n) v - nu u (grad v . n)
//   B(v, lam) = int_dK (c- - pen) lam v + nu lam (grad v . n)
//   C(mu, u)  = int_dK -(c+ + pen) u mu + nu (grad u . n) mu
//   D(mu, lam)= int_dK -(c- - pen) lam mu  (+ c+ lam mu on Neumann facets)
//   F(v)      = int_K f v,   G(mu) = int_{dK on Neumann} g mu, g = -a_hat_n u0 where a_hat_n < 0
// (grad and grad . n spatial).  The Dirichlet trace is the L2 projection of
// the data onto the facet basis and moves to the right-hand side.
//
// One warp per element: the local matrices live in shared memory, lanes run
// over matrix entries (each summing over the quadrature points) and over the
// rows / columns of the elimination.  Then one lane per free facet sums the
// two diagonal contributions in element order and inverts the diagonal block
// by Gauss-Jordan, and one warp per free facet scales its rows.  FP64 throughout.
//
// What bounds it: FP64 issue.  GB300 has two FP64 lanes per SM and clock, so
// one FP64 warp instruction holds an SM for 16 cycles whatever number of its
// lanes work, and loads, index arithmetic and shuffles hide behind it.  The
// kernels are therefore arranged for few, full FP64 instructions:
//  - geometry, normals and the perm of every facet are computed by one thread
//    per element (geometry_kernel) instead of by all 32 lanes of its warp;
//  - products that entries share are computed once per point, and products
//    with components of a gradient that are zero everywhere not at all;
//  - C is built facet by facet after the solve, and its product with the
//    solution goes straight to the rows of the system;
//  - the velocity gradient forms A alone, its constant parts from reference
//    integrals, and sums everything else over the points.
// hdg_element_kernel, 82,944 elements, D = 3, p = 2: 24.7 ms; 29,478
// elements, p = 3: 49.0 ms (65.1 and 133.7 ms with every entry on its own).  The
// FP64 instructions alone take about 21 and 44 ms.
#include <math.h>

#include "air_internal.cuh"
#include "lane_dense.cuh"

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int WPB = 4;         // elements (warps) per block
constexpr int FWPB = 4;        // facets (warps) per block of facet_scale_kernel
constexpr int8_t K_DIR = 1, K_NEU = 2;

__host__ __device__ constexpr int binom(int n, int k) { return k == 0 ? 1 : binom(n - 1, k - 1) * n / k; }
__host__ __device__ constexpr int ipow(int b, int e) { return e == 0 ? 1 : b * ipow(b, e - 1); }
__host__ __device__ constexpr int fact(int n) { return n <= 1 ? 1 : n * fact(n - 1); }

template <int D, int P>
struct Dims {
    static constexpr int NB = binom(P + D, D);       // element basis
    static constexpr int B = binom(P + D - 1, D - 1); // trace basis per facet
    static constexpr int NF = D + 1;
    static constexpr int NT = NF * B;
    static constexpr int NX = NT + 1;                // columns of [B | F]
    static constexpr int Q = P + 2;
    static constexpr int NQ = ipow(Q, D);
    static constexpr int NQF = ipow(Q, D - 1);
    static constexpr int NPERM = fact(D);
    static constexpr int NS = NB * (NB + 1) / 2;     // entries i <= j of a symmetric element matrix
    static constexpr int MAXN = 2 * D;               // off-diagonal facet blocks per row
    // geometry record of an element: J^-1, |det J|, pen, the spatial metric, then per facet the normal, the surface
    // factor and J^-1 (0, n)
    static constexpr int G_DET = D * D, G_PEN = G_DET + 1, G_MM = G_PEN + 1, G_F = G_MM + D * D, G_FS = 2 * D + 1;
    static constexpr int GEO = G_F + NF * G_FS;
    // shared memory of a warp (doubles): A; [B | F], first the volume points; products of one chunk of points, later
    // C and S of one facet; facet point weights; D of one facet; F; the geometry record
    static constexpr int QV = 8, QC = 16;            // volume and facet points per chunk
    static constexpr int XR = NB * NX > NQ * (D + 2) ? NB * NX : NQ * (D + 2);
    static constexpr int PV = QV * NB * (1 + D * D), PF = 4 * QC * NB, PS = NB * B + B * NX;
    static constexpr int PR = PV > PF ? (PV > PS ? PV : PS) : (PF > PS ? PF : PS);
    static constexpr int WARP_DOUBLES = NB * NB + XR + PR + 4 * NF * NQF + B * B + NB + GEO;
    // gradient: A, volume points, chunk products, facet point weights, two facet fields, Lam, mu, U, y, F, geometry
    static constexpr int GRAD_DOUBLES =
        NB * NB + NQ * (D + 1) + QC * NB + 4 * NF * NQF + 2 * NT + 3 * NB + GEO;
    // reference integrals (doubles): volume stiffness per metric entry k <= l, then per facet and frame the
    // symmetrised trace-gradient matrix
    static constexpr int NM = D * (D + 1) / 2;
    static constexpr int T_L = NM * NS, TABLE = T_L + NF * NPERM * D * NS;
};

// (i, j), i <= j, of entry t of a symmetric n x n matrix stored by rows
__device__ __forceinline__ void sym_entry(int t, int n, int &i, int &j) {
    i = 0;
    while (t >= n - i) { t -= n - i; ++i; }
    j = i + t;
}

template <int D>
struct Geo {
    double X0[D];
    double J[D][D];      // J[r][c] = X_{c+1}[r] - X_0[r]
    double Jinv[D][D];
    double det;          // |det J|
    double h;            // longest edge
};

template <int D>
__device__ void geometry(const double *verts, const int32_t *ev, Geo<D> &g) {
    double X[D + 1][D];
#pragma unroll
    for (int v = 0; v <= D; ++v)
#pragma unroll
        for (int d = 0; d < D; ++d) X[v][d] = verts[(int64_t)ev[v] * D + d];
#pragma unroll
    for (int d = 0; d < D; ++d) g.X0[d] = X[0][d];
#pragma unroll
    for (int r = 0; r < D; ++r)
#pragma unroll
        for (int c = 0; c < D; ++c) g.J[r][c] = X[c + 1][r] - X[0][r];
    double det;
    if constexpr (D == 2) {
        det = g.J[0][0] * g.J[1][1] - g.J[0][1] * g.J[1][0];
        g.Jinv[0][0] = g.J[1][1] / det;
        g.Jinv[0][1] = -g.J[0][1] / det;
        g.Jinv[1][0] = -g.J[1][0] / det;
        g.Jinv[1][1] = g.J[0][0] / det;
    } else {
        const double(*J)[D] = g.J;
        double c00 = J[1][1] * J[2][2] - J[1][2] * J[2][1];
        double c01 = J[1][2] * J[2][0] - J[1][0] * J[2][2];
        double c02 = J[1][0] * J[2][1] - J[1][1] * J[2][0];
        det = J[0][0] * c00 + J[0][1] * c01 + J[0][2] * c02;
        g.Jinv[0][0] = c00 / det;
        g.Jinv[1][0] = c01 / det;
        g.Jinv[2][0] = c02 / det;
        g.Jinv[0][1] = (J[0][2] * J[2][1] - J[0][1] * J[2][2]) / det;
        g.Jinv[1][1] = (J[0][0] * J[2][2] - J[0][2] * J[2][0]) / det;
        g.Jinv[2][1] = (J[0][1] * J[2][0] - J[0][0] * J[2][1]) / det;
        g.Jinv[0][2] = (J[0][1] * J[1][2] - J[0][2] * J[1][1]) / det;
        g.Jinv[1][2] = (J[0][2] * J[1][0] - J[0][0] * J[1][2]) / det;
        g.Jinv[2][2] = (J[0][0] * J[1][1] - J[0][1] * J[1][0]) / det;
    }
    g.det = fabs(det);
    double h = 0.0;
#pragma unroll
    for (int i = 0; i <= D; ++i)
#pragma unroll
        for (int j = i + 1; j <= D; ++j) {
            double s = 0.0;
#pragma unroll
            for (int d = 0; d < D; ++d) s += (X[i][d] - X[j][d]) * (X[i][d] - X[j][d]);
            h = fmax(h, sqrt(s));
        }
    g.h = h;
}

// Index s of the canonical frame of local facet k: the facet's local vertices
// (ascending local index) sorted by global id; perms[s] lists, for canonical
// vertex m, the position within the local list.
template <int D>
__device__ int facet_perm(const int32_t *ev, int k, const int32_t *perms) {
    int loc[D], ord[D];
    int32_t gid[D];
    int c = 0;
#pragma unroll
    for (int v = 0; v <= D; ++v)
        if (v != k) loc[c++] = v;
#pragma unroll
    for (int m = 0; m < D; ++m) {
        gid[m] = ev[loc[m]];
        ord[m] = m;
    }
    for (int i = 1; i < D; ++i)          // stable insertion sort of positions by global id
        for (int j = i; j > 0 && gid[ord[j - 1]] > gid[ord[j]]; --j) {
            int t = ord[j];
            ord[j] = ord[j - 1];
            ord[j - 1] = t;
        }
    for (int s = 0; s < fact(D); ++s) {
        bool eq = true;
#pragma unroll
        for (int m = 0; m < D; ++m) eq = eq && perms[s * D + m] == ord[m];
        if (eq) return s;
    }
    return 0;
}

struct ElemArgs {
    int64_t E;
    double nu, alpha;
    int dlen;                    // stored entries of a diagonal row block: 1 (scaled) or b
    const double *verts;
    const int32_t *elems, *elem_facets, *facet_elems;
    const int8_t *kind;
    const int32_t *rnum, *nbr, *nbr_cnt;
    const int64_t *row_ptr;
    const double *wq, *phi, *gphi, *wf, *psi, *phi_f, *gphi_f;
    const int32_t *perms;
    const double *geo, *table;          // E geometry records, reference integrals
    const int32_t *order, *gmask;       // entries of A in the order the lanes take them, components of each gradient
    const int32_t *frame;               // E x NF: canonical frame of the facet, + 256 on Neumann facets
    const double *vel_vol, *src, *vel_face, *u0_face, *lam_dir;
    double *val, *dpart, *hpart;
    // velocity gradient (adjoint) mode
    const double *lam_full, *mu_full;   // n_facets x b trace and unscaled adjoint (0 on Dirichlet)
    double *grad;                       // E x (D-1)
    int *err;
};

// gmask[i]: bit k set when component k of grad phi_i is not zero at every volume point.  order: the entries (i, j) of
// A by falling number of products d_k phi_i d_l phi_j, so that a warp's lanes have equally many.  One thread block.
template <int D, int P>
__device__ void order_entries(const double *gphi, int32_t *order, int32_t *gmask) {
    using Dm = Dims<D, P>;
    constexpr int NB = Dm::NB, NV = Dm::NQ * NB * D;
    __shared__ int mask[NB];
    __shared__ uint8_t products[NB * NB];
    for (int i = threadIdx.x; i < NB; i += blockDim.x) mask[i] = 0;
    __syncthreads();
#pragma unroll 8
    for (int t = threadIdx.x; t < NV; t += blockDim.x)
        if (gphi[t] != 0.0) atomicOr(&mask[t / D % NB], 1 << t % D);
    __syncthreads();
    for (int i = threadIdx.x; i < NB; i += blockDim.x) gmask[i] = mask[i];
    for (int t = threadIdx.x; t < NB * NB; t += blockDim.x)
        products[t] = (uint8_t)(__popc(mask[t / NB]) * __popc(mask[t % NB]));
    __syncthreads();
    for (int t = threadIdx.x; t < NB * NB; t += blockDim.x) {
        const int mine = products[t];
        int place = 0;
#pragma unroll 8
        for (int u = 0; u < NB * NB; ++u) place += products[u] > mine || (products[u] == mine && u < t) ? 1 : 0;
        order[place] = t;
    }
}

// Geometry record and facet frames of every element, one thread per element; with `order` the last block orders the
// entries of A instead (a launch less on small meshes, which are bound by launches).
template <int D, int P>
__global__ void __launch_bounds__(128) geometry_kernel(ElemArgs a, double *geo, int32_t *frame, int32_t *order) {
    using Dm = Dims<D, P>;
    constexpr int NF = Dm::NF;
    if (order && blockIdx.x == gridDim.x - 1) {
        order_entries<D, P>(a.gphi, order, order + Dm::NB * Dm::NB);
        return;
    }
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= a.E) return;
    const int32_t *ev = a.elems + e * (D + 1);
    Geo<D> g;
    geometry<D>(a.verts, ev, g);
    double *o = geo + e * Dm::GEO;
#pragma unroll
    for (int k = 0; k < D; ++k)
#pragma unroll
        for (int d = 0; d < D; ++d) o[k * D + d] = g.Jinv[k][d];
    o[Dm::G_DET] = g.det;
    o[Dm::G_PEN] = __ddiv_rn(__dmul_rn(a.nu, a.alpha), g.h);
#pragma unroll
    for (int k = 0; k < D; ++k)      // spatial metric: sum over spatial s of Jinv[k][s] Jinv[l][s]
#pragma unroll
        for (int l = 0; l < D; ++l) {
            double s = __dmul_rn(g.Jinv[k][1], g.Jinv[l][1]);
            if (D == 3)
                s = k == l ? __fma_rn(g.Jinv[k][1], g.Jinv[k][1], __dmul_rn(g.Jinv[k][D - 1], g.Jinv[k][D - 1]))
                           : __fma_rn(g.Jinv[k][D - 1], g.Jinv[l][D - 1], s);
            o[Dm::G_MM + k * D + l] = s;
        }
#pragma unroll
    for (int k = 0; k < NF; ++k) {
        double gl[D];   // Jinv^T grad_ref(lambda_k): lambda_0 = 1 - sum xi, lambda_k = xi_{k-1}
#pragma unroll
        for (int d = 0; d < D; ++d) {
            if (k == 0) {
                double sum = 0.0;
#pragma unroll
                for (int kk = 0; kk < D; ++kk) sum -= g.Jinv[kk][d];
                gl[d] = sum;
            } else {
                gl[d] = g.Jinv[k > 0 ? k - 1 : 0][d];
            }
        }
        double gn = __fma_rn(gl[0], gl[0], __dmul_rn(gl[1], gl[1]));
        if (D == 3) gn = __fma_rn(gl[D - 1], gl[D - 1], gn);
        gn = sqrt(gn);
        double *f = o + Dm::G_F + k * Dm::G_FS;
        double nh[D];
#pragma unroll
        for (int d = 0; d < D; ++d) f[d] = nh[d] = __ddiv_rn(-gl[d], gn);      // outward unit space-time normal
        const double ws = __dmul_rn(__dmul_rn(__dmul_rn((double)D, __ddiv_rn(g.det, (double)fact(D))), gn), (double)fact(D - 1));
        f[D] = ws;
#pragma unroll
        for (int kk = 0; kk < D; ++kk) {    // (grad phi . n) = grad_ref phi . (Jinv (0, n))
            double sum = __dmul_rn(g.Jinv[kk][1], nh[1]);
            if (D == 3) sum = __fma_rn(g.Jinv[kk][D - 1], nh[D - 1], sum);
            f[D + 1 + kk] = sum;
        }
        frame[e * NF + k] =
            facet_perm<D>(ev, k, a.perms) + (a.kind[a.elem_facets[e * NF + k]] == K_NEU ? 256 : 0);
    }
}

// Reference integrals, one thread each: sum_q wq (d_k phi_i d_l phi_j + d_l phi_i d_k phi_j, or once when k = l)
// and, per facet and frame, sum_q wf (phi_i d_d phi_j + d_d phi_i phi_j).
template <int D, int P>
__global__ void table_kernel(const double *wq, const double *gphi, const double *wf, const double *phi_f,
                             const double *gphi_f, double *table) {
    using Dm = Dims<D, P>;
    constexpr int NB = Dm::NB, NS = Dm::NS;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= Dm::TABLE) return;
    double acc = 0.0;
    if (t < Dm::T_L) {
        int k, l, i, j;
        sym_entry(t / NS, D, k, l);
        sym_entry(t % NS, NB, i, j);
        for (int q = 0; q < Dm::NQ; ++q) {
            const double *gi = gphi + (q * NB + i) * D, *gj = gphi + (q * NB + j) * D;
            acc += wq[q] * (k == l ? gi[k] * gj[k] : gi[k] * gj[l] + gi[l] * gj[k]);
        }
    } else {
        const int u = t - Dm::T_L, ks = u / (D * NS), d = u / NS % D;
        int i, j;
        sym_entry(u % NS, NB, i, j);
        for (int q = 0; q < Dm::NQF; ++q) {
            const int fi = (ks * Dm::NQF + q) * NB + i, fj = (ks * Dm::NQF + q) * NB + j;
            acc += wf[q] * (phi_f[fi] * gphi_f[fj * D + d] + gphi_f[fi * D + d] * phi_f[fj]);
        }
    }
    table[t] = acc;
}

// Volume part: sA = - sum_q W phi_j a_hat.grad_hat phi_i, sF = sum_q W f phi_i.  sV (NQ (D + 1)) and sP are scratch;
// sV keeps -W Jinv a_hat of every point, and W f after them.
template <int D, int P>
__device__ __forceinline__ void volume_part(const ElemArgs &a, int64_t e, const double *sGeo, double *sA, double *sV,
                                            double *sP, double *sF) {
    using Dm = Dims<D, P>;
    constexpr int NB = Dm::NB, NQ = Dm::NQ, QC = Dm::QC, R = (NB * NB + 31) / 32;
    const int lane = threadIdx.x & 31;
    for (int q = lane; q < NQ; q += 32) {
        const double W = sGeo[Dm::G_DET] * a.wq[q];
#pragma unroll
        for (int k = 0; k < D; ++k) {
            double at = sGeo[k * D];
#pragma unroll
            for (int m = 0; m < D - 1; ++m) at += sGeo[k * D + m + 1] * a.vel_vol[(e * NQ + q) * (D - 1) + m];
            sV[q * D + k] = -W * at;
        }
        sV[NQ * D + q] = a.src ? W * a.src[e * NQ + q] : 0.0;
    }
    __syncwarp();
    {   // F: lane groups over the points of one basis function
        constexpr int GR = 32 / NB;
        const int g = lane / NB, i = lane % NB;
        double f = 0.0;
        if (g < GR)
            for (int q = g; q < NQ; q += GR) f += sV[NQ * D + q] * a.phi[q * NB + i];
        double s = f;
#pragma unroll
        for (int k = 1; k < GR; ++k) s += __shfl_sync(FULL, f, (lane + k * NB) & 31);
        if (lane < NB) sF[lane] = s;
    }
    double acc[R];
    int oi[R], oj[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int t = lane + 32 * r < NB * NB ? lane + 32 * r : 0;
        acc[r] = 0.0;
        oi[r] = t / NB;
        oj[r] = t % NB;
    }
    for (int q0 = 0; q0 < NQ; q0 += QC) {
        const int nq = NQ - q0 < QC ? NQ - q0 : QC;
        __syncwarp();
        for (int t = lane; t < nq * NB; t += 32) {
            const int q = q0 + t / NB;
            const double *gp = a.gphi + (q0 * NB + t) * D;
            double adv = 0.0;
#pragma unroll
            for (int k = 0; k < D; ++k) adv += sV[q * D + k] * gp[k];
            sP[t] = adv;
        }
        __syncwarp();
        const double *ph = a.phi + q0 * NB;
        double part[R];                              // a chunk's sum first: shorter chains of roundings
#pragma unroll
        for (int r = 0; r < R; ++r) part[r] = 0.0;
#pragma unroll 4
        for (int q = 0; q < nq; ++q)
#pragma unroll
            for (int r = 0; r < R; ++r) part[r] += sP[q * NB + oi[r]] * ph[q * NB + oj[r]];
#pragma unroll
        for (int r = 0; r < R; ++r) acc[r] += part[r];
    }
    __syncwarp();
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (lane + 32 * r < NB * NB) sA[lane + 32 * r] = acc[r];
}

// Weights of every facet point: W (c+ + pen) and W (c- - pen).
template <int D, int P>
__device__ __forceinline__ void facet_points(const ElemArgs &a, int64_t e, const double *sGeo, double *sW) {
    using Dm = Dims<D, P>;
    constexpr int NF = Dm::NF, NQF = Dm::NQF;
    const double pen = sGeo[Dm::G_PEN];
    for (int t = threadIdx.x & 31; t < NF * NQF; t += 32) {
        const int k = t / NQF, q = t % NQF;
        const double *f = sGeo + Dm::G_F + k * Dm::G_FS;
        double an = f[0];
#pragma unroll
        for (int m = 0; m < D - 1; ++m) an += a.vel_face[((e * NF + k) * NQF + q) * (D - 1) + m] * f[m + 1];
        const double W = f[D] * a.wf[q], cup = 0.5 * (an + fabs(an)), cdn = 0.5 * (an - fabs(an));
        sW[2 * t] = W * (cup + pen);
        sW[2 * t + 1] = W * (cdn - pen);
    }
}

// sP[q NB + i] = w(q) phi_i(q) for one chunk of a facet's points (w every other double from sw).
template <int NB>
__device__ __forceinline__ void weigh(const double *sw, const double *ph, int nq, double *sP) {
    __syncwarp();
    for (int t = threadIdx.x & 31; t < nq * NB; t += 32) sP[t] = sw[2 * (t / NB)] * ph[t];
    __syncwarp();
}

// Adds the diffusion and facet parts of A (all symmetric) to sA.
template <int D, int P>
__device__ __forceinline__ void symmetric_part(const ElemArgs &a, const double *sGeo, const int32_t *fr,
                                               const double *sW, double *sP, double *sA) {
    using Dm = Dims<D, P>;
    constexpr int NB = Dm::NB, NF = Dm::NF, NQF = Dm::NQF, QC = Dm::QC, NS = Dm::NS, R = (NS + 31) / 32;
    const int lane = threadIdx.x & 31;
    const bool diff = a.nu != 0.0;
    double acc[R];
    int ot[R], oi[R], oj[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        ot[r] = lane + 32 * r < NS ? lane + 32 * r : 0;
        sym_entry(ot[r], NB, oi[r], oj[r]);
        acc[r] = 0.0;
        if (diff) {
            int m = 0;
#pragma unroll
            for (int k = 0; k < D; ++k)
#pragma unroll
                for (int l = k; l < D; ++l) acc[r] += sGeo[Dm::G_MM + k * D + l] * a.table[m++ * NS + ot[r]];
            acc[r] *= a.nu * sGeo[Dm::G_DET];
        }
    }
    for (int k = 0; k < NF; ++k) {
        const int ks = k * Dm::NPERM + (fr[k] & 255);
        const double *ph = a.phi_f + (size_t)ks * NQF * NB;
#pragma unroll 1
        for (int q0 = 0; q0 < NQF; q0 += QC) {
            const int nq = NQF - q0 < QC ? NQF - q0 : QC;
            weigh<NB>(sW + 2 * (k * NQF + q0), ph + q0 * NB, nq, sP);
            double part[R];
#pragma unroll
            for (int r = 0; r < R; ++r) part[r] = 0.0;
#pragma unroll 4
            for (int q = 0; q < nq; ++q)
#pragma unroll
                for (int r = 0; r < R; ++r) part[r] += sP[q * NB + oi[r]] * ph[(q0 + q) * NB + oj[r]];
#pragma unroll
            for (int r = 0; r < R; ++r) acc[r] += part[r];
        }
        if (diff) {
            const double *L = a.table + Dm::T_L + (size_t)ks * D * NS;
#pragma unroll
            for (int d = 0; d < D; ++d) {
                const double nj = a.nu * sGeo[Dm::G_F + k * Dm::G_FS + D] * sGeo[Dm::G_F + k * Dm::G_FS + D + 1 + d];
#pragma unroll
                for (int r = 0; r < R; ++r) acc[r] -= nj * L[d * NS + ot[r]];
            }
        }
    }
    __syncwarp();
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (lane + 32 * r < NS) {
            sA[oi[r] * NB + oj[r]] += acc[r];
            if (oi[r] != oj[r]) sA[oj[r] * NB + oi[r]] += acc[r];
        }
    __syncwarp();
}

// LU factors of the warp's A (N x N, row-major) with partial pivoting (ties -> smallest row), the row operations
// applied to the NC columns of X (row stride LDX) on the way; the multipliers stay below the diagonal, perm (registers,
// lane c < N) gets the row swapped with row c.  Returns false if a pivot is zero.
template <int N, int NC, int LDX>
__device__ bool warp_factor(double *A, double *X, int &perm) {
    const int lane = threadIdx.x & 31;
    perm = lane;
    for (int c = 0; c < N; ++c) {
        unsigned long long v = 0ull;
        int r = N;
        const int rr0 = c + lane;                    // N <= 32: one row per lane
        if (rr0 < N) {
            v = magnitude_key(A[rr0 * N + c]);
            r = rr0;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long ov = __shfl_xor_sync(FULL, v, o);
            const int orow = __shfl_xor_sync(FULL, r, o);
            if (ov > v || (ov == v && orow < r)) { v = ov; r = orow; }
        }
        if (v <= 1ull) return false;                 // zero, or nothing but NaN
        if (lane == c) perm = r;
        if (r != c) {
            for (int t = lane; t < N + NC; t += 32) {
                double *u = t < N ? A + c * N + t : X + c * LDX + (t - N), *w = t < N ? A + r * N + t : X + r * LDX + (t - N);
                const double x = *u;
                *u = *w;
                *w = x;
            }
            __syncwarp();
        }
        if (rr0 > c && rr0 < N) A[rr0 * N + c] = A[rr0 * N + c] / A[c * N + c];
        __syncwarp();
        const int wa = N - c - 1, w = wa + NC;
        if (w > 0) {
            int rr = c + 1 + lane / w, cc = lane % w;
            while (rr < N) {
                const double m = A[rr * N + c];
                if (cc < wa) A[rr * N + c + 1 + cc] -= m * A[c * N + c + 1 + cc];
                else X[rr * LDX + (cc - wa)] -= m * X[c * LDX + (cc - wa)];
                cc += 32;
                while (cc >= w) { cc -= w; ++rr; }
            }
        }
        __syncwarp();
    }
    return true;
}

// X <- U^{-1} X for the factors of warp_factor, row by row from the last
template <int N, int NC, int LDX>
__device__ void warp_back_substitute(const double *A, double *X) {
    const int lane = threadIdx.x & 31;
    for (int r = N - 1; r >= 0; --r) {
        for (int t = lane; t < NC; t += 32) X[r * LDX + t] = X[r * LDX + t] / A[r * N + r];
        __syncwarp();
        for (int t = lane; t < r * NC; t += 32) {
            const int rr = t / NC, cc = t % NC;
            X[rr * LDX + cc] -= A[rr * N + r] * X[r * LDX + cc];
        }
        __syncwarp();
    }
}

// The assembled system keeps the bits it had when every entry was evaluated on
// its own.  That is a choice: solutions and V-cycles of an FP32 hierarchy stay
// comparable bit by bit between versions.  Accuracy does not ask for it: with the
// sums rearranged freely the entries' error against 64 bits was the same, one
// FP32 V-cycle moved by 1.6e-9 (its own error is 2e-7), and the assembly took 8.9
// and 14.6 ms instead of 27.0 (82,944 elements, p = 2) and 51.1 ms (29,478
// elements, p = 3).  So every entry is
// evaluated with the operations of its plain expression (in the comments below),
// written as intrinsics, and summed over the points in their order.  Which of an
// entry's products are fused differs with D and P (the conditions on them
// below); it was found by comparing outputs with the plain form and means nothing
// in the mathematics.  What entries share
// (products of one point's weight with one basis function, the gradient in the
// flow's direction) is computed once and kept in shared memory, and terms
// that vanish for every point (a monomial's gradient has few components) are
// left out of a sum, which changes nothing.

// Volume part of A and F:
//   A(i, j) = sum_q W ( -phi_j adv_i + nu sum_kl Mm_kl d_k phi_i d_l phi_j ),  adv_i = (Jinv a_hat) . grad phi_i
//   F(i)    = sum_q (W f) phi_i
// sV: W, Jinv a_hat and W f of every point.  sP: adv_i and Mm_kl d_k phi_i of one chunk of points.
template <int D, int P>
__device__ __forceinline__ void exact_volume(const ElemArgs &a, int64_t e, const double *sGeo, double *sA, double *sV,
                                             double *sP, double *sF) {
    using Dm = Dims<D, P>;
    constexpr int NB = Dm::NB, NQ = Dm::NQ, QV = Dm::QV, R = (NB * NB + 31) / 32, DD = D * D;
    const int lane = threadIdx.x & 31;
    const bool diff = a.nu != 0.0;
    double *sT = sV + NQ, *sS = sT + NQ * D, *sM = sP + QV * NB;
    for (int q = lane; q < NQ; q += 32) {
        const double W = __dmul_rn(sGeo[Dm::G_DET], a.wq[q]);
        sV[q] = W;
#pragma unroll
        for (int k = 0; k < D; ++k) {
            double at = sGeo[k * D];
#pragma unroll
            for (int m = 0; m < D - 1; ++m) at = __fma_rn(sGeo[k * D + m + 1], a.vel_vol[(e * NQ + q) * (D - 1) + m], at);
            sT[q * D + k] = at;
        }
        sS[q] = a.src ? __dmul_rn(W, a.src[e * NQ + q]) : 0.0;
    }
    __syncwarp();
    for (int i = lane; i < NB; i += 32) {
        double f = 0.0;
        if (a.src)
            for (int q = 0; q < NQ; ++q) f = __fma_rn(sS[q], a.phi[q * NB + i], f);
        sF[i] = f;
    }
    // the lane's entries, those with equally many diffusion terms together
    double acc[R];
    int oi[R], oj[R], mi[R], mj[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int t = a.order[lane + 32 * r < NB * NB ? lane + 32 * r : NB * NB - 1];
        acc[r] = 0.0;
        oi[r] = t / NB;
        oj[r] = t % NB;
        mi[r] = diff ? a.gmask[oi[r]] : 0;
        mj[r] = diff ? a.gmask[oj[r]] : 0;
    }
    for (int q0 = 0; q0 < NQ; q0 += QV) {
        const int nq = NQ - q0 < QV ? NQ - q0 : QV;
        __syncwarp();
        for (int t = lane; t < nq * NB; t += 32) {
            const int q = q0 + t / NB;
            const double *gp = a.gphi + (q0 * NB + t) * D;
            double adv = __dmul_rn(sT[q * D], gp[0]);
#pragma unroll
            for (int k = 1; k < D; ++k) adv = __fma_rn(sT[q * D + k], gp[k], adv);
            sP[t] = adv;
        }
        if (diff)
            for (int t = lane; t < nq * NB * DD; t += 32)
                sM[t] = __dmul_rn(sGeo[Dm::G_MM + t % DD], a.gphi[q0 * NB * D + t / D]);
        __syncwarp();
        const double *ph = a.phi + q0 * NB, *gq = a.gphi + q0 * NB * D;
#pragma unroll 1
        for (int q = 0; q < nq; ++q) {
            const double W = sV[q0 + q];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                double term = __dmul_rn(-ph[q * NB + oj[r]], sP[q * NB + oi[r]]);
                int m1 = mi[r], m2 = mj[r];
                if (m1 && m2) {
                    const double *pm = sM + (q * NB + oi[r]) * DD, *gj = gq + (q * NB + oj[r]) * D;
                    double dif = 0.0;
                    do {                             // components k of grad phi_i, l of grad phi_j, ascending
                        const int k = __ffs(m1) - 1, l = __ffs(m2) - 1;
                        dif = __fma_rn(pm[k * D + l], gj[l], dif);
                        m2 &= m2 - 1;
                        if (!m2) {
                            m1 &= m1 - 1;
                            m2 = mj[r];
                        }
                    } while (m1);
                    term = __fma_rn(a.nu, dif, term);
                }
                acc[r] = __fma_rn(W, term, acc[r]);
            }
        }
    }
    __syncwarp();
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (lane + 32 * r < NB * NB) sA[oi[r] * NB + oj[r]] = acc[r];
}

// W, c+, c- and W g of every facet point
template <int D, int P>
__device__ __forceinline__ void exact_facet_points(const ElemArgs &a, int64_t e, const double *sGeo, const int32_t *fr,
                                                   double *sW) {
    using Dm = Dims<D, P>;
    constexpr int NF = Dm::NF, NQF = Dm::NQF;
    for (int t = threadIdx.x & 31; t < NF * NQF; t += 32) {
        const int k = t / NQF, q = t % NQF;
        const double *f = sGeo + Dm::G_F + k * Dm::G_FS;
        double an = f[0];
        const double *vel = a.vel_face + ((e * NF + k) * NQF + q) * (D - 1);
        an = __dadd_rn(an, __dmul_rn(vel[0], f[1]));
        if (D == 3) an = __fma_rn(vel[D - 2], f[D - 1], an);
        const double W = __dmul_rn(f[D], a.wf[q]);
        sW[4 * t] = W;
        sW[4 * t + 1] = __dmul_rn(0.5, __dadd_rn(an, fabs(an)));
        sW[4 * t + 2] = __dmul_rn(0.5, __dsub_rn(an, fabs(an)));
        double gN = 0.0;
        if (fr[k] >= 256 && an < 0.0 && a.u0_face) gN = __dmul_rn(-an, a.u0_face[(e * NF + k) * NQF + q]);
        sW[4 * t + 3] = __dmul_rn(W, gN);
    }
}

// Products of one chunk of facet points with every basis function: (c+ + pen) phi, (c- - pen) phi, grad phi . n and nu
// times it, each nq x NB.
template <int D, int P>
__device__ __forceinline__ void exact_facet_products(const ElemArgs &a, const double *sGeo, int k, int ks, int q0,
                                                     int nq, const double *sW, double *sP) {
    using Dm = Dims<D, P>;
    constexpr int NB = Dm::NB, NQF = Dm::NQF, N = Dm::QC * NB;
    const double *f = sGeo + Dm::G_F + k * Dm::G_FS + D + 1, pen = sGeo[Dm::G_PEN];
    __syncwarp();
    for (int t = threadIdx.x & 31; t < nq * NB; t += 32) {
        const int q = q0 + t / NB;
        const size_t at = ((size_t)ks * NQF + q0) * NB + t;
        const double fi = a.phi_f[at], cup = sW[4 * (k * NQF + q) + 1], cdn = sW[4 * (k * NQF + q) + 2];
        sP[t] = __dmul_rn(__dadd_rn(cup, pen), fi);
        sP[N + t] = __dmul_rn(__dsub_rn(cdn, pen), fi);
        double dn = __dmul_rn(a.gphi_f[at * D], f[0]);
#pragma unroll
        for (int d = 1; d < D; ++d) dn = __fma_rn(a.gphi_f[at * D + d], f[d], dn);
        sP[2 * N + t] = dn;
        sP[3 * N + t] = __dmul_rn(a.nu, dn);
    }
    __syncwarp();
}

// Facet k's parts of A and B:
//   A(i, j) += sum_q W ( (c+ + pen) phi_i phi_j - nu (phi_i dn_j + dn_i phi_j) )
//   B(i, m)  = sum_q W ( (c- - pen) phi_i psi_m + nu dn_i psi_m )
template <int D, int P>
__device__ __forceinline__ void exact_facet(const ElemArgs &a, const double *sGeo, int k, int ks, const double *sW,
                                            double *sP, double *sA, double *sX) {
    using Dm = Dims<D, P>;
    constexpr int NB = Dm::NB, B = Dm::B, NX = Dm::NX, NQF = Dm::NQF, QC = Dm::QC, N = QC * NB,
                  R = (NB * NB + 31) / 32, RB = (NB * B + 31) / 32;
    const int lane = threadIdx.x & 31;
    const bool diff = a.nu != 0.0;
    double acc[R], bcc[RB];
    int oi[R], oj[R], bi[RB], bm[RB];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int t = lane + 32 * r < NB * NB ? lane + 32 * r : 0;
        acc[r] = 0.0;
        oi[r] = t / NB;
        oj[r] = t % NB;
    }
#pragma unroll
    for (int r = 0; r < RB; ++r) {
        const int t = lane + 32 * r < NB * B ? lane + 32 * r : 0;
        bcc[r] = 0.0;
        bi[r] = t / B;
        bm[r] = t % B;
    }
#pragma unroll 1
    for (int q0 = 0; q0 < NQF; q0 += QC) {
        const int nq = NQF - q0 < QC ? NQF - q0 : QC;
        exact_facet_products<D, P>(a, sGeo, k, ks, q0, nq, sW, sP);
        const double *ph = a.phi_f + ((size_t)ks * NQF + q0) * NB, *ps = a.psi + q0 * B;
#pragma unroll 1
        for (int q = 0; q < nq; ++q) {
            const double W = sW[4 * (k * NQF + q0 + q)];
            const double *p = sP + q * NB, *f = ph + q * NB;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int i = oi[r], j = oj[r];
                double term = __dmul_rn(p[i], f[j]);
                if (diff) {
                    const double cross = __fma_rn(p[2 * N + i], f[j], __dmul_rn(f[i], p[2 * N + j]));
                    term = P > 1 ? __fma_rn(p[i], f[j], -__dmul_rn(a.nu, cross)) : __fma_rn(-a.nu, cross, term);
                }
                acc[r] = __fma_rn(W, term, acc[r]);
            }
#pragma unroll
            for (int r = 0; r < RB; ++r) {
                const double pl = ps[q * B + bm[r]];
                double term = __dmul_rn(p[N + bi[r]], pl);
                if (diff)
                    term = D + P > 4 ? __fma_rn(p[N + bi[r]], pl, __dmul_rn(p[3 * N + bi[r]], pl))
                                     : __fma_rn(p[3 * N + bi[r]], pl, term);
                bcc[r] = __fma_rn(W, term, bcc[r]);
            }
        }
    }
    __syncwarp();
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (lane + 32 * r < NB * NB) sA[lane + 32 * r] = __dadd_rn(sA[lane + 32 * r], acc[r]);
#pragma unroll
    for (int r = 0; r < RB; ++r)
        if (lane + 32 * r < NB * B) sX[bi[r] * NX + k * B + bm[r]] = bcc[r];
}

// Facet k's C, transposed (j, m) in sP:  C(m, j) = sum_q W ( -(c+ + pen) phi_j psi_m + nu dn_j psi_m )
template <int D, int P>
__device__ __forceinline__ void exact_coupling(const ElemArgs &a, const double *sGeo, int k, int ks, const double *sW,
                                               double *sP) {
    using Dm = Dims<D, P>;
    constexpr int NB = Dm::NB, B = Dm::B, NQF = Dm::NQF, QC = Dm::QC, N = QC * NB, RB = (NB * B + 31) / 32;
    const int lane = threadIdx.x & 31;
    const bool diff = a.nu != 0.0;
    double acc[RB];
    int oj[RB], om[RB];
#pragma unroll
    for (int r = 0; r < RB; ++r) {
        const int t = lane + 32 * r < NB * B ? lane + 32 * r : 0;
        acc[r] = 0.0;
        oj[r] = t / B;
        om[r] = t % B;
    }
#pragma unroll 1
    for (int q0 = 0; q0 < NQF; q0 += QC) {
        const int nq = NQF - q0 < QC ? NQF - q0 : QC;
        exact_facet_products<D, P>(a, sGeo, k, ks, q0, nq, sW, sP);
        const double *ps = a.psi + q0 * B;
#pragma unroll 2
        for (int q = 0; q < nq; ++q) {
            const double W = sW[4 * (k * NQF + q0 + q)];
#pragma unroll
            for (int r = 0; r < RB; ++r) {
                const double pl = ps[q * B + om[r]];
                double term = __dmul_rn(-sP[q * NB + oj[r]], pl);
                if (diff) term = __fma_rn(sP[3 * N + q * NB + oj[r]], pl, term);
                acc[r] = __fma_rn(W, term, acc[r]);
            }
        }
    }
    __syncwarp();
#pragma unroll
    for (int r = 0; r < RB; ++r)
        if (lane + 32 * r < NB * B) sP[lane + 32 * r] = acc[r];
}

// Gaussian elimination with partial pivoting (ties -> smallest row) of the warp's A (N x N, row-major) applied to the
// NC columns of X (row stride LDX), then back substitution column by column: X <- A^{-1} X.  Returns false if a pivot
// is zero.
template <int N, int NC, int LDX>
__device__ bool warp_solve(double *A, double *X) {
    const int lane = threadIdx.x & 31;
    for (int c = 0; c < N; ++c) {
        unsigned long long v = 0ull;
        int r = N;
        const int rr0 = c + lane;                    // N <= 32: one row per lane
        if (rr0 < N) {
            v = magnitude_key(A[rr0 * N + c]);
            r = rr0;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long ov = __shfl_xor_sync(FULL, v, o);
            const int orow = __shfl_xor_sync(FULL, r, o);
            if (ov > v || (ov == v && orow < r)) { v = ov; r = orow; }
        }
        if (v <= 1ull) return false;                 // zero, or nothing but NaN
        if (r != c) {
            for (int t = lane; t < N + NC; t += 32) {
                double *u = t < N ? A + c * N + t : X + c * LDX + (t - N), *w = t < N ? A + r * N + t : X + r * LDX + (t - N);
                const double x = *u;
                *u = *w;
                *w = x;
            }
            __syncwarp();
        }
        if (rr0 > c && rr0 < N) A[rr0 * N + c] = __ddiv_rn(A[rr0 * N + c], A[c * N + c]);
        __syncwarp();
        const int wa = N - c - 1, w = wa + NC;
        int rr = c + 1 + lane / w, cc = lane % w;
        while (rr < N) {
            const double m = A[rr * N + c];
            if (cc < wa) A[rr * N + c + 1 + cc] = __fma_rn(-m, A[c * N + c + 1 + cc], A[rr * N + c + 1 + cc]);
            else X[rr * LDX + (cc - wa)] = __fma_rn(-m, X[c * LDX + (cc - wa)], X[rr * LDX + (cc - wa)]);
            cc += 32;
            while (cc >= w) { cc -= w; ++rr; }
        }
        __syncwarp();
    }
    for (int t = lane; t < NC; t += 32)
        for (int r = N - 1; r >= 0; --r) {
            double s = X[r * LDX + t];
            for (int cc = r + 1; cc < N; ++cc) s = __fma_rn(-A[r * N + cc], X[cc * LDX + t], s);
            X[r * LDX + t] = __ddiv_rn(s, A[r * N + r]);
        }
    __syncwarp();
    return true;
}

template <int D, int P>
__global__ void __launch_bounds__(WPB * 32) hdg_element_kernel(ElemArgs a) {
    using Dm = Dims<D, P>;
    constexpr int NB = Dm::NB, B = Dm::B, NF = Dm::NF, NT = Dm::NT, NX = Dm::NX, MAXN = Dm::MAXN, NQF = Dm::NQF;
    extern __shared__ double smem[];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t e = (int64_t)blockIdx.x * WPB + w;
    if (e >= a.E) return;                                 // the whole warp leaves together
    double *sA = smem + (size_t)w * Dm::WARP_DOUBLES;
    double *sX = sA + NB * NB, *sP = sX + Dm::XR, *sW = sP + Dm::PR, *sD = sW + 4 * NF * NQF, *sF = sD + B * B,
           *sGeo = sF + NB;
    const int32_t *fr = a.frame + e * NF, *ef = a.elem_facets + e * NF;
    for (int t = lane; t < Dm::GEO; t += 32) sGeo[t] = a.geo[e * Dm::GEO + t];
    __syncwarp();
    exact_volume<D, P>(a, e, sGeo, sA, sX, sP, sF);
    exact_facet_points<D, P>(a, e, sGeo, fr, sW);
    for (int k = 0; k < NF; ++k) exact_facet<D, P>(a, sGeo, k, k * Dm::NPERM + (fr[k] & 255), sW, sP, sA, sX);
    for (int i = lane; i < NB; i += 32) sX[i * NX + NT] = sF[i];
    __syncwarp();
    if (!warp_solve<NB, NX, NX>(sA, sX)) {
        if (lane == 0) atomicOr(a.err, AIR_DEVERR_SINGULAR);
        return;
    }
    // rows of facet k: S_k = D_k - C_k X_B and H_k = G_k - C_k X_F - sum over Dirichlet facets l of S_kl Lam_l
    for (int k = 0; k < NF; ++k) {
        const int32_t f = ef[k];
        if (a.kind[f] == K_DIR) continue;
        exact_coupling<D, P>(a, sGeo, k, k * Dm::NPERM + (fr[k] & 255), sW, sP);
        const double pen = sGeo[Dm::G_PEN];
        for (int t = lane; t < B * B; t += 32) {      // D(m, l) = sum_q W ( -(c- - pen) (+ c+) ) psi_l psi_m
            const int m = t / B, l = t % B;
            double s = 0.0;
            for (int q = 0; q < NQF; ++q) {
                const double *p = sW + 4 * (k * NQF + q);
                const double wc = __dmul_rn(p[0], __dadd_rn(-__dsub_rn(p[2], pen), fr[k] >= 256 ? p[1] : 0.0));
                s = __fma_rn(__dmul_rn(wc, a.psi[q * B + l]), a.psi[q * B + m], s);
            }
            sD[t] = s;
        }
        double g = 0.0;
        if (lane < B)
            for (int q = 0; q < NQF; ++q) g = __fma_rn(sW[4 * (k * NQF + q) + 3], a.psi[q * B + lane], g);
        const int slot = a.facet_elems[2 * (int64_t)f] == (int32_t)e ? 0 : 1;
        const int32_t rf = a.rnum[f];
        // lane l: where block (k, l) starts within a row, -1 when it is not stored
        int off = -1;
        if (lane < NF && lane != k && a.kind[ef[lane]] != K_DIR) {
            const int cnt = a.nbr_cnt[rf];
            const int32_t *nb = a.nbr + (int64_t)rf * MAXN;
            const int32_t rg = a.rnum[ef[lane]];
            int rank = 0;
            while (rank < cnt && nb[rank] != rg) ++rank;
            if (rank == cnt) atomicOr(a.err, AIR_DEVERR_CSR);
            else off = rank * B + (rg > rf ? a.dlen : 0);
        }
        const int64_t row0 = a.row_ptr[(int64_t)rf * B], rowlen = a.row_ptr[(int64_t)rf * B + 1] - row0;
        double *dp = a.dpart + (2 * (int64_t)f + slot) * B * B, *sS = sP + NB * B;
        __syncwarp();
#pragma unroll 2
        for (int t0 = 0; t0 < B * NX; t0 += 32) {
            const int t = t0 + lane < B * NX ? t0 + lane : 0;
            const int m = t / NX, c = t % NX, l = c / B;
            double s = 0.0;
#pragma unroll
            for (int i = 0; i < NB; ++i) s = __fma_rn(sP[i * B + m], sX[i * NX + c], s);
            const int o = __shfl_sync(FULL, off, l & 31);
            const double gm = __shfl_sync(FULL, g, m);
            if (t0 + lane >= B * NX) continue;
            const double v = __dsub_rn(c == NT ? gm : (l == k ? sD[m * B + c - k * B] : 0.0), s);
            sS[t] = v;
            if (l == k) dp[m * B + c - k * B] = v;
            else if (o >= 0) a.val[row0 + m * rowlen + o + c - l * B] = v;
        }
        __syncwarp();
        for (int m = lane; m < B; m += 32) {
            double h = sS[m * NX + NT];
            for (int l = 0; l < NF; ++l) {
                if (l == k || a.kind[ef[l]] != K_DIR) continue;
                const double *ld = a.lam_dir + (int64_t)ef[l] * B;
                for (int l2 = 0; l2 < B; ++l2) h = __fma_rn(-sS[m * NX + l * B + l2], ld[l2], h);
            }
            a.hpart[(2 * (int64_t)f + slot) * B + m] = h;
        }
        __syncwarp();
    }
}

// ---------------------------------------------------------------- pattern
__global__ void free_flag_kernel(int64_t F, const int8_t *kind, int32_t *flag) {
    for (int64_t f = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; f < F; f += (int64_t)gridDim.x * blockDim.x)
        flag[f] = kind[f] != K_DIR ? 1 : 0;
}

__global__ void renumber_kernel(int64_t F, const int8_t *kind, const int64_t *scan, int32_t *rnum,
                                int32_t *free_ids) {
    for (int64_t f = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; f < F; f += (int64_t)gridDim.x * blockDim.x) {
        if (kind[f] != K_DIR) {
            rnum[f] = (int32_t)scan[f];
            free_ids[scan[f]] = (int32_t)f;
        } else {
            rnum[f] = -1;
        }
    }
}

// Sorted free neighbour facets (by free number) of every free facet: the
// other facets of its one or two elements.
template <int D>
__global__ void neighbour_kernel(int64_t nfree, int B, int dlen, const int32_t *free_ids, const int32_t *facet_elems,
                                 const int32_t *elem_facets, const int8_t *kind, const int32_t *rnum, int32_t *nbr,
                                 int32_t *cnt, int32_t *rowlen) {
    constexpr int MAXN = 2 * D;
    for (int64_t rf = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; rf < nfree;
         rf += (int64_t)gridDim.x * blockDim.x) {
        const int32_t f = free_ids[rf];
        int32_t list[MAXN];
        int c = 0;
        for (int s = 0; s < 2; ++s) {
            const int32_t e = facet_elems[2 * (int64_t)f + s];
            if (e < 0) continue;
            for (int l = 0; l <= D; ++l) {
                const int32_t g = elem_facets[(int64_t)e * (D + 1) + l];
                if (g == f || kind[g] == K_DIR || c >= MAXN) continue;
                int32_t v = rnum[g];
                int j = c++;
                while (j > 0 && list[j - 1] > v) { list[j] = list[j - 1]; --j; }
                list[j] = v;
            }
        }
        for (int t = 0; t < MAXN; ++t) nbr[rf * MAXN + t] = t < c ? list[t] : -1;
        cnt[rf] = c;
        for (int i = 0; i < B; ++i) rowlen[rf * B + i] = c * B + dlen;
    }
}

template <int MAXN>
__global__ void columns_kernel(int64_t nfree, int B, int dlen, const int32_t *nbr, const int32_t *cnt,
                               const int64_t *row_ptr, int32_t *col) {
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < nfree * B;
         r += (int64_t)gridDim.x * blockDim.x) {
        const int64_t rf = r / B;
        const int i = (int)(r % B);
        const int c = cnt[rf];
        int64_t p = row_ptr[r];
        bool diag = false;
        for (int t = 0; t <= c; ++t) {
            const int32_t g = t < c ? nbr[rf * MAXN + t] : INT32_MAX;
            if (!diag && g > rf) {
                diag = true;
                if (dlen == 1) col[p++] = (int32_t)(rf * B + i);
                else for (int j = 0; j < B; ++j) col[p++] = (int32_t)(rf * B + j);
            }
            if (t < c)
                for (int j = 0; j < B; ++j) col[p++] = g * B + j;
        }
    }
}

__global__ void dirichlet_kernel(int64_t F, int B, int NQF, const int8_t *kind, const double *proj, const double *gd,
                                 double *lam) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < F * B; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t f = t / B;
        const int m = (int)(t % B);
        double s = 0.0;
        if (kind[f] == K_DIR && gd)
            for (int q = 0; q < NQF; ++q) s += proj[m * NQF + q] * gd[f * NQF + q];
        lam[t] = s;
    }
}

struct FacetArgs {
    int64_t nfree;
    int B, dlen, maxn, scale;
    const int32_t *free_ids, *facet_elems, *nbr, *cnt;
    const int64_t *row_ptr;
    const double *hpart;
    double *dpart;               // two b x b slots per facet; the first then takes the inverse
    double *val, *rhs, *diag;
    int *err;
};

// Sd = sum of the element contributions (element order) of every free facet,
// one facet per lane: written to diag, and inverted into the facet's first
// slot of dpart (scaled) or written to the diagonal blocks of its rows.
// With facet_scale_kernel it takes 1.0 ms for 57,222 facets of 10 unknowns
// (2.1 ms with the inverse by one warp per facet), 0.7 ms for 164,736 facets of
// 6 (2.8 ms).
__global__ void __launch_bounds__(32) facet_block_kernel(FacetArgs a) {
    extern __shared__ double smem[];
    const int lane = threadIdx.x, B = a.B, BB = B * B;
    const int64_t first = (int64_t)blockIdx.x * 32;
    const int count = a.nfree - first < 32 ? (int)(a.nfree - first) : 32;
    for (int k = 0; k < count; ++k) {
        const int32_t f = a.free_ids[first + k];
        const bool two = a.facet_elems[2 * (int64_t)f + 1] >= 0;
        const int64_t rf = first + k, row0 = a.row_ptr[rf * B], len = a.row_ptr[rf * B + 1] - row0;
        int64_t at = 0;
        if (!a.scale)
            for (int t = 0; t < a.cnt[rf]; ++t) at += a.nbr[rf * a.maxn + t] < rf ? B : 0;
        for (int t = lane; t < BB; t += 32) {
            double v = a.dpart[(2 * (int64_t)f) * BB + t];
            if (two) v = v + a.dpart[(2 * (int64_t)f + 1) * BB + t];
            smem[t * LANE_LD + k] = v;
            if (a.diag) a.diag[rf * BB + t] = v;
            if (!a.scale) a.val[row0 + (t / B) * len + at + t % B] = v;
        }
    }
    if (!a.scale) return;
    __syncwarp();
    if (lane < count && !lane_invert(smem + lane, B)) atomicOr(a.err, AIR_DEVERR_SINGULAR);
    __syncwarp();
    for (int k = 0; k < count; ++k) {
        const int64_t f = a.free_ids[first + k];
        for (int t = lane; t < BB; t += 32) a.dpart[2 * f * BB + t] = smem[t * LANE_LD + k];
    }
}

// One warp per free facet: its b rows, all of one length, are read as one
// run, multiplied by the inverse of the diagonal block and written back; H
// takes the diagonal's column, whose product is the right-hand side, and the
// diagonal itself is stored as ones.  Unscaled: rhs = H alone.
__global__ void __launch_bounds__(FWPB * 32) facet_scale_kernel(FacetArgs a) {
    extern __shared__ double smem[];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, B = a.B;
    const int64_t rf = (int64_t)blockIdx.x * FWPB + w;
    if (rf >= a.nfree) return;
    const int64_t f = a.free_ids[rf];
    const bool two = a.facet_elems[2 * f + 1] >= 0;
    double *sI = smem + (size_t)w * (B * B + B * (a.maxn * B + 1)), *sT = sI + B * B;
    const int64_t row0 = a.row_ptr[rf * B];
    const int len = (int)(a.row_ptr[rf * B + 1] - row0), c = a.cnt[rf];
    int at = 0;                                       // the diagonal's place in a row
    for (int t = 0; t < c; ++t) at += a.nbr[rf * a.maxn + t] < rf ? B : 0;
    for (int m = lane; m < B; m += 32) {
        double h = a.hpart[2 * f * B + m];
        if (two) h = h + a.hpart[(2 * f + 1) * B + m];
        if (a.scale) sT[m * len + at] = h;
        else a.rhs[rf * B + m] = h;
    }
    if (!a.scale) return;
    for (int t = lane; t < B * B; t += 32) sI[t] = a.dpart[2 * f * B * B + t];
    for (int t = lane; t < B * len; t += 32)
        if (t % len != at) sT[t] = a.val[row0 + t];
    __syncwarp();
    for (int t = lane; t < B * len; t += 32) {
        const int m = t / len, l = t % len;
        double s = 0.0;
        for (int j = 0; j < B; ++j) s += sI[m * B + j] * sT[j * len + l];
        a.val[row0 + t] = l == at ? 1.0 : s;
        if (l == at) a.rhs[rf * B + m] = s;
    }
}

// --------------------------------------------------------------- points
template <int D>
__global__ void points_kernel(int64_t E, int nq, int nqf, int nperm, const double *verts, const int32_t *elems,
                              const double *xq, const double *xi_f, const int32_t *perms, double *x_vol,
                              double *x_face) {
    const int64_t per = (int64_t)nq + (int64_t)(D + 1) * nqf;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < E * per;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = t / per;
        const int r = (int)(t % per);
        const int32_t *ev = elems + e * (D + 1);
        double X0[D], J[D][D];
#pragma unroll
        for (int d = 0; d < D; ++d) X0[d] = verts[(int64_t)ev[0] * D + d];
#pragma unroll
        for (int d = 0; d < D; ++d)
#pragma unroll
            for (int c = 0; c < D; ++c) J[d][c] = verts[(int64_t)ev[c + 1] * D + d] - X0[d];
        const double *xi;
        double *out;
        if (r < nq) {
            if (!x_vol) continue;
            xi = xq + r * D;
            out = x_vol + (e * nq + r) * D;
        } else {
            if (!x_face) continue;
            const int k = (r - nq) / nqf, q = (r - nq) % nqf;
            const int s = facet_perm<D>(ev, k, perms);
            xi = xi_f + ((int64_t)(k * nperm + s) * nqf + q) * D;
            out = x_face + ((e * (D + 1) + k) * nqf + q) * D;
        }
#pragma unroll
        for (int d = 0; d < D; ++d) {
            double v = X0[d];
#pragma unroll
            for (int c = 0; c < D; ++c) v += J[d][c] * xi[c];
            out[d] = v;
        }
    }
}

__global__ void facet_points_kernel(int64_t F, int D, int nqf, const double *verts, const int32_t *facets,
                                    const double *sq, double *x_facet) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < F * nqf;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t f = t / nqf;
        const int q = (int)(t % nqf);
        const int32_t *fv = facets + f * D;
        for (int d = 0; d < D; ++d) {
            const double w0 = verts[(int64_t)fv[0] * D + d];
            double v = w0;
            for (int m = 0; m + 1 < D; ++m) v += (verts[(int64_t)fv[m + 1] * D + d] - w0) * sq[q * (D - 1) + m];
            x_facet[t * D + d] = v;
        }
    }
}

// ------------------------------------------------------ velocity gradient
// mu_f = Sd_f^{-T} adj_f per free facet (the unscaled adjoint), spread to all
// facets with zeros on Dirichlet ones; Lambda likewise with the Dirichlet
// values.  One facet per lane.
__global__ void __launch_bounds__(32) adjoint_unscale_kernel(int64_t nfree, int B, const int32_t *free_ids,
                                                             const double *diag, const double *lam,
                                                             const double *adj, double *mu_full, double *lam_full,
                                                             int *err) {
    extern __shared__ double smem[];
    const int lane = threadIdx.x;
    const int64_t first = (int64_t)blockIdx.x * 32;
    const int count = nfree - first < 32 ? (int)(nfree - first) : 32;
    double *sx = smem + B * B * LANE_LD;
    lane_load_blocks(diag, first, count, B, true, smem);
    for (int t = lane; t < count * B; t += 32) sx[(t % B) * LANE_LD + t / B] = adj[first * B + t];
    __syncwarp();
    if (lane < count && !lane_invert(smem + lane, B)) atomicOr(err, AIR_DEVERR_SINGULAR);
    __syncwarp();
    for (int t = lane; t < count * B; t += 32) {
        const int k = t / B, i = t % B;
        double v = 0.0;
        for (int j = 0; j < B; ++j) v += smem[(i * B + j) * LANE_LD + k] * sx[j * LANE_LD + k];
        const int64_t o = (int64_t)free_ids[first + k] * B + i;
        mu_full[o] = v;
        lam_full[o] = lam[first * B + t];
    }
}

__global__ void spread_dirichlet_kernel(int64_t F, int B, const int8_t *kind, const double *lam_dir, double *mu_full,
                                        double *lam_full) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < F * B; t += (int64_t)gridDim.x * blockDim.x)
        if (kind[t / B] == K_DIR) {
            mu_full[t] = 0.0;
            lam_full[t] = lam_dir[t];
        }
}

// dL/da_e,m = mu^T (dH/da - dS/da Lambda) = -mu^T dC U + y^T dA U - mu^T dD Lambda + y^T dB Lambda
// with U = A^{-1}(F - B Lambda), y = A^{-T} C^T mu (the source and the
// Neumann data do not depend on the element velocity here: on the t faces the
// spatial normal vanishes).  Only A is formed: B Lambda and C^T mu are sums
// over the facet points with the fields Lambda and mu there, one
// factorisation serves both solves, and with u = U phi, y = y phi, lam and mu
// at the points the derivative is
//   sum_facet W n_m [ (1 + s)/2 (y u + u mu - neu lam mu) + (1 - s)/2 (y lam + lam mu) ]
//   - sum_volume W (Jinv e_m).grad_hat(y) u,    s = sign(a_hat_n), 0 on the kink.
// 48,000 elements, D = 3, p = 2: 3.7 ms (61.9 ms when A, B, C, D and their
// derivatives were formed and two factorisations made).
template <int D, int P>
__global__ void __launch_bounds__(WPB * 32) velocity_gradient_kernel(ElemArgs a) {
    using Dm = Dims<D, P>;
    constexpr int NB = Dm::NB, B = Dm::B, NF = Dm::NF, NT = Dm::NT, NQ = Dm::NQ, NQF = Dm::NQF;
    extern __shared__ double smem[];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t e = (int64_t)blockIdx.x * WPB + w;
    if (e >= a.E) return;
    double *sA = smem + (size_t)w * Dm::GRAD_DOUBLES;
    double *sV = sA + NB * NB, *sP = sV + NQ * (D + 1), *sW = sP + Dm::QC * NB, *sL = sW + 2 * NF * NQF,
           *sM = sL + NF * NQF, *sLam = sM + NF * NQF, *sMu = sLam + NT, *sU = sMu + NT, *sY = sU + NB, *sF = sY + NB,
           *sGeo = sF + NB;
    const int32_t *fr = a.frame + e * NF, *ef = a.elem_facets + e * NF;
    for (int t = lane; t < Dm::GEO; t += 32) sGeo[t] = a.geo[e * Dm::GEO + t];
    for (int t = lane; t < NT; t += 32) {
        const int k = t / B, m = t % B;
        sLam[t] = a.lam_full[(int64_t)ef[k] * B + m];
        sMu[t] = a.mu_full[(int64_t)ef[k] * B + m];
    }
    __syncwarp();
    volume_part<D, P>(a, e, sGeo, sA, sV, sP, sF);
    facet_points<D, P>(a, e, sGeo, sW);
    symmetric_part<D, P>(a, sGeo, fr, sW, sP, sA);
    for (int t = lane; t < NF * NQF; t += 32) {
        const int k = t / NQF, q = t % NQF;
        double l = 0.0, u = 0.0;
#pragma unroll
        for (int m = 0; m < B; ++m) {
            l += a.psi[q * B + m] * sLam[k * B + m];
            u += a.psi[q * B + m] * sMu[k * B + m];
        }
        sL[t] = l;
        sM[t] = u;
    }
    __syncwarp();
    {   // F - B Lam and C^T mu: lane groups over the facet points of one basis function
        constexpr int GR = 32 / NB;
        const int g = lane / NB, i = lane % NB;
        double bl = 0.0, cm = 0.0;
        if (g < GR)
            for (int t = g; t < NF * NQF; t += GR) {
                const int k = t / NQF, q = t % NQF;
                const size_t at = ((size_t)(k * Dm::NPERM + (fr[k] & 255)) * NQF + q) * NB + i;
                const double f = a.phi_f[at];
                bl += sW[2 * t + 1] * sL[t] * f;
                cm -= sW[2 * t] * sM[t] * f;
                if (a.nu != 0.0) {
                    double dn = 0.0;
#pragma unroll
                    for (int d = 0; d < D; ++d) dn += sGeo[Dm::G_F + k * Dm::G_FS + D + 1 + d] * a.gphi_f[at * D + d];
                    dn *= a.nu * sGeo[Dm::G_F + k * Dm::G_FS + D] * a.wf[q];
                    bl += dn * sL[t];
                    cm += dn * sM[t];
                }
            }
        double s1 = bl, s2 = cm;
#pragma unroll
        for (int k = 1; k < GR; ++k) {
            s1 += __shfl_sync(FULL, bl, (lane + k * NB) & 31);
            s2 += __shfl_sync(FULL, cm, (lane + k * NB) & 31);
        }
        if (lane < NB) {
            sU[lane] = sF[lane] - s1;
            sY[lane] = s2;
        }
    }
    __syncwarp();
    int perm;
    if (!warp_factor<NB, 1, 1>(sA, sU, perm)) {
        if (lane == 0) atomicOr(a.err, AIR_DEVERR_SINGULAR);
        return;
    }
    warp_back_substitute<NB, 1, 1>(sA, sU);
    // A^T y = c: U^T z = c, L^T v = z, then the row swaps undone in reverse
    double y = lane < NB ? sY[lane] : 0.0;
    for (int c = 0; c < NB; ++c) {
        const double z = __shfl_sync(FULL, y, c) / sA[c * NB + c];
        if (lane == c) y = z;
        if (lane > c && lane < NB) y -= sA[c * NB + lane] * z;
    }
    for (int c = NB - 1; c > 0; --c) {
        const double z = __shfl_sync(FULL, y, c);
        if (lane < c) y -= sA[c * NB + lane] * z;
    }
    for (int c = NB - 1; c >= 0; --c) {
        const int r = __shfl_sync(FULL, perm, c);
        const double yc = __shfl_sync(FULL, y, c), yr = __shfl_sync(FULL, y, r);
        if (lane == c) y = yr;
        else if (lane == r) y = yc;
    }
    if (lane < NB) sY[lane] = y;
    __syncwarp();
    double part[D - 1];
#pragma unroll
    for (int m = 0; m < D - 1; ++m) part[m] = 0.0;
    for (int t = lane; t < NF * NQF; t += 32) {
        const int k = t / NQF, q = t % NQF;
        const double *f = sGeo + Dm::G_F + k * Dm::G_FS;
        const double *ph = a.phi_f + ((size_t)(k * Dm::NPERM + (fr[k] & 255)) * NQF + q) * NB;
        double u = 0.0, v = 0.0;
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            u += ph[i] * sU[i];
            v += ph[i] * sY[i];
        }
        double an = f[0];
#pragma unroll
        for (int m = 0; m < D - 1; ++m) an += a.vel_face[((e * NF + k) * NQF + q) * (D - 1) + m] * f[m + 1];
        const double s = an > 0.0 ? 1.0 : (an < 0.0 ? -1.0 : 0.0), l = sL[t], mu = sM[t];
        const double up = v * u + u * mu - (fr[k] >= 256 ? l * mu : 0.0), dn = v * l + l * mu;
        const double wv = f[D] * a.wf[q] * (0.5 * (1.0 + s) * up + 0.5 * (1.0 - s) * dn);
#pragma unroll
        for (int m = 0; m < D - 1; ++m) part[m] += wv * f[m + 1];
    }
    for (int q = lane; q < NQ; q += 32) {
        double u = 0.0, gy[D];
#pragma unroll
        for (int d = 0; d < D; ++d) gy[d] = 0.0;
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            u += a.phi[q * NB + i] * sU[i];
#pragma unroll
            for (int d = 0; d < D; ++d) gy[d] += a.gphi[(q * NB + i) * D + d] * sY[i];
        }
        const double wu = sGeo[Dm::G_DET] * a.wq[q] * u;
#pragma unroll
        for (int m = 0; m < D - 1; ++m) {
            double t = 0.0;
#pragma unroll
            for (int d = 0; d < D; ++d) t += sGeo[d * D + m + 1] * gy[d];
            part[m] -= wu * t;
        }
    }
#pragma unroll
    for (int m = 0; m < D - 1; ++m) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) part[m] += __shfl_down_sync(FULL, part[m], o);
        if (lane == 0) a.grad[e * (D - 1) + m] = part[m];
    }
}

// ---------------------------------------------------------------- host side
unsigned grid_for(int64_t items, int threads) {
    int64_t b = (items + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > 152 * 32) b = 152 * 32;
    return (unsigned)b;
}

int check_ref(const air_hdg_mesh *M, const air_hdg_ref *R) {
    if (!M || !R || (M->D != 2 && M->D != 3) || R->p < 1 || R->p > 3) return AIR_ERR_INVALID_ARG;
    const int D = M->D, p = R->p, q = p + 2;
    if (R->nb != binom(p + D, D) || R->b != binom(p + D - 1, D - 1) || R->nq != ipow(q, D) ||
        R->nqf != ipow(q, D - 1) || R->nperm != fact(D))
        return AIR_ERR_INVALID_ARG;
    if (M->n_elems <= 0 || M->n_facets <= 0 || M->n_verts <= 0 || !M->verts || !M->elems || !M->elem_facets ||
        !M->facets || !M->facet_elems || !M->facet_kind)
        return AIR_ERR_INVALID_ARG;
    if (M->n_elems > INT32_MAX || M->n_facets > INT32_MAX) return AIR_ERR_INVALID_ARG;
    return AIR_OK;
}

template <typename T>
int dalloc(T **p, int64_t count) {
    *p = nullptr;
    if (count <= 0) count = 1;
    AIR_CUDA(air_dmalloc((void **)p, (size_t)count * sizeof(T)));
    return AIR_OK;
}

// Facet renumbering and the neighbour lists (the pattern of every row).
struct Pattern {
    int64_t nfree = 0, nnz = 0;
    int32_t *rnum = nullptr, *free_ids = nullptr, *nbr = nullptr, *cnt = nullptr, *rowlen = nullptr;
    int64_t *scan = nullptr;
    ~Pattern() {
        air_dfree(rnum); air_dfree(free_ids); air_dfree(nbr); air_dfree(cnt); air_dfree(rowlen); air_dfree(scan);
    }
};

int build_pattern(const air_hdg_mesh *M, const air_hdg_ref *R, int dlen, int64_t *row_ptr, Pattern &P,
                  cudaStream_t s) {
    const int64_t F = M->n_facets;
    const int D = M->D, B = R->b, MAXN = 2 * D;
    int32_t *flag = nullptr;
    AIR_TRY(dalloc(&flag, F));
    AIR_TRY(dalloc(&P.scan, F + 1));
    free_flag_kernel<<<air_counted(grid_for(F, 256)), 256, 0, s>>>(F, M->facet_kind, flag);
    AIR_LAUNCH();
    int st = air_exclusive_scan_i32(flag, P.scan, F, s);
    air_dfree(flag);
    AIR_TRY(st);
    AIR_CUDA(cudaMemcpyAsync(&P.nfree, P.scan + F, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    AIR_CUDA(cudaStreamSynchronize(s));
    AIR_TRY(dalloc(&P.rnum, F));
    AIR_TRY(dalloc(&P.free_ids, P.nfree));
    renumber_kernel<<<air_counted(grid_for(F, 256)), 256, 0, s>>>(F, M->facet_kind, P.scan, P.rnum, P.free_ids);
    AIR_LAUNCH();
    AIR_TRY(dalloc(&P.nbr, P.nfree * MAXN));
    AIR_TRY(dalloc(&P.cnt, P.nfree));
    AIR_TRY(dalloc(&P.rowlen, P.nfree * B));
    if (D == 2)
        neighbour_kernel<2><<<air_counted(grid_for(P.nfree, 256)), 256, 0, s>>>(
            P.nfree, B, dlen, P.free_ids, M->facet_elems, M->elem_facets, M->facet_kind, P.rnum, P.nbr, P.cnt,
            P.rowlen);
    else
        neighbour_kernel<3><<<air_counted(grid_for(P.nfree, 256)), 256, 0, s>>>(
            P.nfree, B, dlen, P.free_ids, M->facet_elems, M->elem_facets, M->facet_kind, P.rnum, P.nbr, P.cnt,
            P.rowlen);
    AIR_LAUNCH();
    int64_t *rp = row_ptr;
    if (!rp) AIR_TRY(dalloc(&rp, P.nfree * B + 1));
    st = air_exclusive_scan_i32(P.rowlen, rp, P.nfree * B, s);
    if (st == AIR_OK) {
        cudaError_t e = cudaMemcpyAsync(&P.nnz, rp + P.nfree * B, sizeof(int64_t), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) st = AIR_ERR_CUDA;
    }
    if (!row_ptr) air_dfree(rp);
    return st;
}

template <int D, int P>
int launch_element(ElemArgs &a, bool gradient, cudaStream_t s) {
    using Dm = Dims<D, P>;
    const size_t smem = (size_t)WPB * (gradient ? Dm::GRAD_DOUBLES : Dm::WARP_DOUBLES) * sizeof(double);
    if (smem > AIR_SMEM_OPTIN) return AIR_ERR_UNSUPPORTED;
    // geometry records, then the gradient's reference integrals; facet frames, then the assembly's order of entries
    double *geo = nullptr;
    int32_t *frame = nullptr;
    int st = dalloc(&geo, a.E * Dm::GEO + (gradient ? Dm::TABLE : 0));
    if (st == AIR_OK) st = dalloc(&frame, a.E * Dm::NF + (gradient ? 0 : Dm::NB * Dm::NB + Dm::NB));
    cudaError_t err = cudaSuccess;
    if (st == AIR_OK) {
        double *table = geo + a.E * Dm::GEO;
        int32_t *order = gradient ? nullptr : frame + a.E * Dm::NF;
        geometry_kernel<D, P><<<air_counted((unsigned)((a.E + 127) / 128 + (gradient ? 0 : 1))), 128, 0, s>>>(a, geo, frame,
                                                                                                          order);
        a.geo = geo;
        a.frame = frame;
        const unsigned grid = (unsigned)((a.E + WPB - 1) / WPB);
        if (gradient) {
            table_kernel<D, P><<<air_counted((Dm::TABLE + 127) / 128), 128, 0, s>>>(a.wq, a.gphi, a.wf, a.phi_f,
                                                                                   a.gphi_f, table);
            a.table = table;
            err = air_smem_optin(velocity_gradient_kernel<D, P>);
            if (err == cudaSuccess) velocity_gradient_kernel<D, P><<<air_counted(grid), WPB * 32, smem, s>>>(a);
        } else {
            a.order = order;
            a.gmask = order + Dm::NB * Dm::NB;
            err = air_smem_optin(hdg_element_kernel<D, P>);
            if (err == cudaSuccess) hdg_element_kernel<D, P><<<air_counted(grid), WPB * 32, smem, s>>>(a);
        }
        if (err == cudaSuccess) err = cudaGetLastError();
        if (err != cudaSuccess) st = AIR_ERR_CUDA;
    }
    air_dfree(geo);
    air_dfree(frame);
    return st;
}

int dispatch_element(int D, int p, ElemArgs &a, bool gradient, cudaStream_t s) {
    switch (D * 10 + p) {
    case 21: return launch_element<2, 1>(a, gradient, s);
    case 22: return launch_element<2, 2>(a, gradient, s);
    case 23: return launch_element<2, 3>(a, gradient, s);
    case 31: return launch_element<3, 1>(a, gradient, s);
    case 32: return launch_element<3, 2>(a, gradient, s);
    case 33: return launch_element<3, 3>(a, gradient, s);
    default: return AIR_ERR_INVALID_ARG;
    }
}

ElemArgs element_args(const air_hdg_mesh *M, const air_hdg_ref *R, const air_hdg_data *d) {
    ElemArgs a{};
    a.E = M->n_elems;
    a.nu = d->nu;
    a.alpha = d->alpha;
    a.verts = M->verts;
    a.elems = M->elems;
    a.elem_facets = M->elem_facets;
    a.facet_elems = M->facet_elems;
    a.kind = M->facet_kind;
    a.wq = R->wq; a.phi = R->phi; a.gphi = R->gphi; a.wf = R->wf; a.psi = R->psi;
    a.phi_f = R->phi_f; a.gphi_f = R->gphi_f; a.perms = R->perms;
    a.vel_vol = d->vel_vol; a.src = d->src; a.vel_face = d->vel_face; a.u0_face = d->u0_face;
    return a;
}

int read_err(int *d_err, cudaStream_t s) {
    int h = 0;
    AIR_CUDA(cudaMemcpyAsync(&h, d_err, sizeof(int), cudaMemcpyDeviceToHost, s));
    AIR_CUDA(cudaStreamSynchronize(s));
    if (h & AIR_DEVERR_SINGULAR) return AIR_ERR_SINGULAR_COARSE;
    if (h & AIR_DEVERR_CSR) return AIR_ERR_CSR_MALFORMED;
    return AIR_OK;
}

int assemble_impl(const air_hdg_mesh *M, const air_hdg_ref *R, const air_hdg_data *d, int scale, int64_t *row_ptr,
                  int32_t *col, double *val, double *rhs, double *diag, double *lam_dir, cudaStream_t s) {
    const int D = M->D, B = R->b, dlen = scale ? 1 : B;
    const int64_t F = M->n_facets;
    Pattern P;
    AIR_TRY(build_pattern(M, R, dlen, row_ptr, P, s));
    if (D == 2)
        columns_kernel<4><<<air_counted(grid_for(P.nfree * B, 256)), 256, 0, s>>>(P.nfree, B, dlen, P.nbr, P.cnt,
                                                                                   row_ptr, col);
    else
        columns_kernel<6><<<air_counted(grid_for(P.nfree * B, 256)), 256, 0, s>>>(P.nfree, B, dlen, P.nbr, P.cnt,
                                                                                   row_ptr, col);
    AIR_LAUNCH();
    double *ld = lam_dir, *dpart = nullptr, *hpart = nullptr;
    int *d_err = nullptr;
    int st = AIR_OK;
    if (!ld) st = dalloc(&ld, F * B);
    if (st == AIR_OK) st = dalloc(&dpart, 2 * F * B * B);
    if (st == AIR_OK) st = dalloc(&hpart, 2 * F * B);
    if (st == AIR_OK) st = dalloc(&d_err, 1);
    if (st == AIR_OK) {
        cudaError_t e = cudaMemsetAsync(d_err, 0, sizeof(int), s);
        if (e != cudaSuccess) st = AIR_ERR_CUDA;
    }
    if (st == AIR_OK) {
        dirichlet_kernel<<<air_counted(grid_for(F * B, 256)), 256, 0, s>>>(F, B, R->nqf, M->facet_kind, R->dir_proj,
                                                                          d->g_dir, ld);
        if (cudaGetLastError() != cudaSuccess) st = AIR_ERR_CUDA;
    }
    if (st == AIR_OK) {
        ElemArgs a = element_args(M, R, d);
        a.dlen = dlen;
        a.rnum = P.rnum; a.nbr = P.nbr; a.nbr_cnt = P.cnt; a.row_ptr = row_ptr;
        a.lam_dir = ld; a.val = val; a.dpart = dpart; a.hpart = hpart; a.err = d_err;
        st = dispatch_element(D, R->p, a, false, s);
    }
    if (st == AIR_OK) {
        FacetArgs fa{};
        fa.nfree = P.nfree; fa.B = B; fa.dlen = dlen; fa.maxn = 2 * D; fa.scale = scale;
        fa.free_ids = P.free_ids; fa.facet_elems = M->facet_elems; fa.nbr = P.nbr; fa.cnt = P.cnt;
        fa.row_ptr = row_ptr; fa.dpart = dpart; fa.hpart = hpart; fa.val = val; fa.rhs = rhs; fa.diag = diag;
        fa.err = d_err;
        facet_block_kernel<<<air_counted((unsigned)((P.nfree + 31) / 32)), 32, B * B * LANE_LD * sizeof(double), s>>>(fa);
        facet_scale_kernel<<<air_counted((unsigned)((P.nfree + FWPB - 1) / FWPB)), FWPB * 32,
                             FWPB * (B * B + B * (2 * D * B + 1)) * sizeof(double), s>>>(fa);
        if (cudaGetLastError() != cudaSuccess) st = AIR_ERR_CUDA;
    }
    if (st == AIR_OK) st = read_err(d_err, s);
    if (!lam_dir) air_dfree(ld);
    air_dfree(dpart);
    air_dfree(hpart);
    air_dfree(d_err);
    return st;
}

}  // namespace

extern "C" {

int air_hdg_points(const air_hdg_mesh *M, const air_hdg_ref *R, double *x_vol, double *x_face, double *x_facet,
                   void *stream) {
    AIR_TRY(check_ref(M, R));
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t E = M->n_elems, F = M->n_facets;
    const int D = M->D;
    if (x_vol || x_face) {
        const int64_t items = E * (R->nq + (int64_t)(D + 1) * R->nqf);
        if (D == 2)
            points_kernel<2><<<air_counted(grid_for(items, 256)), 256, 0, s>>>(E, R->nq, R->nqf, R->nperm, M->verts,
                                                                               M->elems, R->xq, R->xi_f, R->perms,
                                                                               x_vol, x_face);
        else
            points_kernel<3><<<air_counted(grid_for(items, 256)), 256, 0, s>>>(E, R->nq, R->nqf, R->nperm, M->verts,
                                                                               M->elems, R->xq, R->xi_f, R->perms,
                                                                               x_vol, x_face);
        AIR_LAUNCH();
    }
    if (x_facet) {
        facet_points_kernel<<<air_counted(grid_for(F * R->nqf, 256)), 256, 0, s>>>(F, D, R->nqf, M->verts, M->facets,
                                                                                   R->sq, x_facet);
        AIR_LAUNCH();
    }
    return AIR_OK;
}

int air_hdg_size(const air_hdg_mesh *M, const air_hdg_ref *R, int scale, int64_t *n_rows, int64_t *nnz,
                 void *stream) {
    AIR_TRY(check_ref(M, R));
    if (!n_rows || !nnz) return AIR_ERR_INVALID_ARG;
    AirCallStream call((cudaStream_t)stream);
    Pattern P;
    AIR_TRY(build_pattern(M, R, scale ? 1 : R->b, nullptr, P, (cudaStream_t)stream));
    *n_rows = P.nfree * R->b;
    *nnz = P.nnz;
    return AIR_OK;
}

int air_hdg_assemble(const air_hdg_mesh *M, const air_hdg_ref *R, const air_hdg_data *data, int scale,
                     int64_t *row_ptr, int32_t *col, double *val, double *rhs, double *diag, double *lam_dir,
                     void *stream) {
    AIR_TRY(check_ref(M, R));
    if (!data || !row_ptr || !col || !val || !rhs || !data->vel_vol || !data->vel_face || !(data->nu >= 0.0))
        return AIR_ERR_INVALID_ARG;
    AirCallStream call((cudaStream_t)stream);
    return assemble_impl(M, R, data, scale ? 1 : 0, row_ptr, col, val, rhs, diag, lam_dir, (cudaStream_t)stream);
}

int air_hdg_velocity_gradient(const air_hdg_mesh *M, const air_hdg_ref *R, const air_hdg_data *data,
                              const double *diag, const double *lam_dir, const double *lam, const double *adj,
                              double *grad, void *stream) {
    AIR_TRY(check_ref(M, R));
    if (!data || !diag || !lam_dir || !lam || !adj || !grad || !data->vel_vol || !data->vel_face)
        return AIR_ERR_INVALID_ARG;
    AirCallStream call((cudaStream_t)stream);
    cudaStream_t s = (cudaStream_t)stream;
    const int D = M->D, B = R->b;
    const int64_t F = M->n_facets;
    Pattern P;
    AIR_TRY(build_pattern(M, R, 1, nullptr, P, s));
    double *mu_full = nullptr, *lam_full = nullptr;
    int *d_err = nullptr;
    int st = dalloc(&mu_full, F * B);
    if (st == AIR_OK) st = dalloc(&lam_full, F * B);
    if (st == AIR_OK) st = dalloc(&d_err, 1);
    if (st == AIR_OK && cudaMemsetAsync(d_err, 0, sizeof(int), s) != cudaSuccess) st = AIR_ERR_CUDA;
    if (st == AIR_OK) {
        adjoint_unscale_kernel<<<air_counted((unsigned)((P.nfree + 31) / 32)), 32,
                                 (B * B + B) * LANE_LD * sizeof(double), s>>>(P.nfree, B, P.free_ids, diag, lam, adj,
                                                                              mu_full, lam_full, d_err);
        spread_dirichlet_kernel<<<air_counted(grid_for(F * B, 256)), 256, 0, s>>>(F, B, M->facet_kind, lam_dir,
                                                                                   mu_full, lam_full);
        if (cudaGetLastError() != cudaSuccess) st = AIR_ERR_CUDA;
    }
    if (st == AIR_OK) {
        ElemArgs a = element_args(M, R, data);
        a.lam_full = lam_full;
        a.mu_full = mu_full;
        a.grad = grad;
        a.err = d_err;
        st = dispatch_element(D, R->p, a, true, s);
    }
    if (st == AIR_OK) st = read_err(d_err, s);
    air_dfree(mu_full);
    air_dfree(lam_full);
    air_dfree(d_err);
    return st;
}

}  // extern "C"
