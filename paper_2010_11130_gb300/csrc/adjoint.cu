// Operations for the adjoint of the condensed system.
//
// A solve u = A^{-1} b of the block-scaled trace system (Section 2.5) has the
// adjoint lambda = A^{-T} g for a loss gradient g = dL/du: then dL/db = lambda
// and dL/da_ij = -lambda_i u_j on the stored entries of A.  A^T keeps the unit
// diagonal blocks of A and is the upwind operator of the reversed flow, so the
// same l-AIR setup applies to it.  This file holds the two operations the
// adjoint needs beyond setup and solve: the transpose of A with its values and
// the outer product restricted to A's pattern.
#include "air_internal.cuh"
#include "lane_dense.cuh"

namespace {

unsigned blocks_for(int64_t items, int threads) {
    int64_t b = (items + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > 152 * 32) b = 152 * 32;
    return (unsigned)b;
}

__global__ void col_count_kernel(int64_t nnz, const int32_t *ci, int64_t ncols, int32_t *cnt, int *err) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nnz; e += (int64_t)gridDim.x * blockDim.x) {
        const int32_t c = ci[e];
        if (c < 0 || c >= ncols) { atomicOr(err, AIR_DEVERR_CSR); continue; }
        atomicAdd(&cnt[c], 1);
    }
}

// Entries of row i go to row ci[e] of the transpose at a claimed slot.
__global__ void scatter_t_kernel(int64_t n, const int64_t *rp, const int32_t *ci, const double *v, int64_t ncols,
                                 const int64_t *rpt, int32_t *fill, int32_t *cit, double *vt) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        for (int64_t e = rp[i]; e < rp[i + 1]; ++e) {
            const int32_t c = ci[e];
            if (c < 0 || c >= ncols) continue;
            const int64_t p = rpt[c] + atomicAdd(&fill[c], 1);
            cit[p] = (int32_t)i;
            vt[p] = v[e];
        }
    }
}

// The slots were claimed in any order: sort each row of the transpose by
// column, one warp per row.  Rows of at most 32 SORT_R entries are held in
// registers (entry lane + 32 r) and every entry's place is the number of
// smaller columns in the row (the columns of a row are distinct; equal ones,
// from a malformed matrix, keep their order); longer rows are sorted in place
// by odd-even transposition.  Bound: the 24 bytes per entry read and written;
// 20.6 M entries, 36 per row: 0.79 ms (one thread per row and an insertion sort
// in global memory: 7.6 ms).
constexpr int SORT_R = 4;

__global__ void __launch_bounds__(256) sort_rows_kernel(int64_t m, const int64_t *rpt, int32_t *cit, double *vt) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; row < m; row += warps) {
        const int64_t b = rpt[row];
        const int64_t len = rpt[row + 1] - b;
        if (len <= 32 * SORT_R) {
            int32_t c[SORT_R];
            double x[SORT_R];
            int place[SORT_R];
#pragma unroll
            for (int r = 0; r < SORT_R; ++r) {
                const bool on = lane + 32 * r < len;
                c[r] = on ? cit[b + lane + 32 * r] : INT32_MAX;
                x[r] = on ? vt[b + lane + 32 * r] : 0.0;
                place[r] = 0;
            }
            __syncwarp();
#pragma unroll
            for (int q = 0; q < SORT_R; ++q) {
                if (32 * q >= len) break;
                const int top = len - 32 * q < 32 ? (int)(len - 32 * q) : 32;
                for (int k = 0; k < top; ++k) {
                    const int32_t o = __shfl_sync(0xffffffffu, c[q], k);
#pragma unroll
                    for (int r = 0; r < SORT_R; ++r)
                        place[r] += o < c[r] || (o == c[r] && k + 32 * q < lane + 32 * r) ? 1 : 0;
                }
            }
#pragma unroll
            for (int r = 0; r < SORT_R; ++r)
                if (lane + 32 * r < len) {
                    cit[b + place[r]] = c[r];
                    vt[b + place[r]] = x[r];
                }
        } else {
            for (int64_t pass = 0; pass < len; ++pass) {
                for (int64_t p = b + (pass & 1) + 2 * lane; p + 1 < b + len; p += 64) {
                    const int32_t c0 = cit[p], c1 = cit[p + 1];
                    if (c0 <= c1) continue;
                    const double x0 = vt[p];
                    cit[p] = c1;
                    cit[p + 1] = c0;
                    vt[p] = vt[p + 1];
                    vt[p + 1] = x0;
                }
                __syncwarp();
            }
        }
    }
}

__global__ void outer_kernel(int64_t n, int64_t ncols, const int64_t *rp, const int32_t *ci, const double *u,
                             const double *w, double alpha, double *out) {
    // one warp per row: u_i once, w gathered along the row
    const int lane = threadIdx.x & 31;
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n; i += warps) {
        const double ai = alpha * u[i];
        for (int64_t e = rp[i] + lane; e < rp[i + 1]; e += 32) {
            const int32_t c = ci[e];
            out[e] = (c >= 0 && c < ncols) ? ai * w[c] : __longlong_as_double(0x7ff8000000000000ll);   // NaN marks a bad column
        }
    }
}

// D_f^{-T} of every facet block, one block per lane.
__global__ void __launch_bounds__(32) invert_transposed_kernel(int64_t nblk, int b, const double *diag, double *inv,
                                                               int *err) {
    extern __shared__ double bsm[];
    const int lane = threadIdx.x, bb = b * b;
    const int64_t first = (int64_t)blockIdx.x * 32;
    const int count = nblk - first < 32 ? (int)(nblk - first) : 32;
    lane_load_blocks(diag, first, count, b, true, bsm);
    if (lane < count && !lane_invert(bsm + lane, b)) atomicOr(err, AIR_DEVERR_SINGULAR);
    __syncwarp();
    for (int k = 0; k < count; ++k)
        for (int t = lane; t < bb; t += 32) inv[(first + k) * bb + t] = bsm[t * LANE_LD + k];
}

// One warp per block row f of A^T (rows f b .. f b + b - 1): every
// off-diagonal block T (columns g b .. g b + b - 1) becomes D_f^{-T} T D_g^T,
// the diagonal block (stored as its b ones) stays the identity.  SCALE_CH
// blocks at a time, so that the two products fill the lanes (FP64 issue bounds
// it; 95,200 rows of 6 x 6 blocks: 0.45 ms, with the inverses 0.6 ms, against
// 3.65 ms for the inverse in the same warp and a product of three factors per
// entry).  Rows of a block row must share one layout of whole blocks;
// otherwise err gets AIR_DEVERR_CSR.
constexpr int SCALE_CH = 6;

__global__ void __launch_bounds__(128) block_scale_t_kernel(int64_t nblk, int b, const double *diag,
                                                            const double *inv, const int64_t *rpt,
                                                            const int32_t *cit, double *vt, int *err) {
    extern __shared__ double bsm[];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t f = (int64_t)blockIdx.x * 4 + w;
    if (f >= nblk) return;
    const int bb = b * b;
    double *Di = bsm + (size_t)w * (1 + 3 * SCALE_CH) * bb, *T = Di + bb, *G = T + SCALE_CH * bb, *Y = G + SCALE_CH * bb;
    const int64_t r0 = f * b, base = rpt[r0];
    const int64_t len = rpt[r0 + 1] - base;
    bool ok = len >= 1 && (len - 1) % b == 0;
    for (int i = 1; i < b && ok; ++i) ok = rpt[r0 + i + 1] - rpt[r0 + i] == len;
    if (!ok) {
        if (lane == 0) atomicOr(err, AIR_DEVERR_CSR);
        return;
    }
    for (int t = lane; t < bb; t += 32) Di[t] = inv[f * bb + t];
    const int64_t nb = (len - 1) / b;
    int64_t p = 0;                      // position within the row
    for (int64_t k0 = 0; k0 < nb; k0 += SCALE_CH) {
        const int ch = nb - k0 < SCALE_CH ? (int)(nb - k0) : SCALE_CH;
        int64_t off[SCALE_CH];          // where the chunk's blocks start: a diagonal entry before one is skipped
        bool good = true;
        for (int k = 0; k < ch; ++k) {
            // nb blocks and one diagonal entry fill the row: a second entry in column block f would overrun it
            if (p < len && cit[base + p] / b == f) ++p;
            if (p + b > len) { good = false; break; }
            off[k] = p;
            p += b;
        }
        for (int k = 0; k < ch && good; ++k) {
            const int32_t cs = cit[base + off[k]];
            const int64_t g = cs / b;
            good = cs % b == 0 && g != f && cs >= 0 && g < nblk;
            for (int t = lane; t < bb && good; t += 32) {
                const int i = t / b, j = t % b;
                good = cit[base + i * len + off[k] + j] == (int32_t)(g * b + j);
                T[k * bb + t] = vt[base + i * len + off[k] + j];
                G[k * bb + t] = diag[g * bb + t];                                     // D_g
            }
            good = __all_sync(0xffffffffu, good);
        }
        if (!good) {
            if (lane == 0) atomicOr(err, AIR_DEVERR_CSR);
            return;
        }
        __syncwarp();
        for (int t = lane; t < ch * bb; t += 32) {            // Y = T D_g^T
            const int k = t / bb, i = t / b % b, j = t % b;
            const double *Tk = T + k * bb + i * b, *Gk = G + k * bb + j * b;
            double acc = 0.0;
            for (int c = 0; c < b; ++c) acc += Tk[c] * Gk[c];
            Y[t] = acc;
        }
        __syncwarp();
        for (int t = lane; t < ch * bb; t += 32) {            // D_f^{-T} Y
            const int k = t / bb, i = t / b % b, j = t % b;
            double acc = 0.0;
            for (int c = 0; c < b; ++c) acc += Di[i * b + c] * Y[k * bb + c * b + j];
            vt[base + i * len + off[k] + j] = acc;
        }
        __syncwarp();
    }
}

// y_k = op(D_k) x_k over the b-blocks: op 0 D, 1 D^T, 2 D^{-1}, 3 D^{-T}.  x is read before y is written, so that they
// may be the same vector.  A group of b lanes per block, a lane per row, 32 / b blocks per warp.  Bound: the blocks'
// bytes without an inverse, FP64 issue with one; whole calls with their synchronisation, blocks of 10: 300,000 of them
// 104 us and 1.05 ms (inverse), 1,000 of them 43 and 62 us.  One block per lane, through shared memory, took 698 us and
// 1.73 ms, 82 and 185 us; one warp per block 266 us and 7.2 ms, 45 and 82 us.
template <bool INVERT>
__global__ void __launch_bounds__(128) block_rows_kernel(int64_t nblk, int b, const double *diag, int op,
                                                         const double *x, double *y, int *err) {
    extern __shared__ double bsm[];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, per = 32 / b, g = lane / b, i = lane % b, bb = b * b;
    const int64_t k = ((int64_t)blockIdx.x * 4 + w) * per + g;
    const bool on = g < per && k < nblk;
    const double *D = diag + (on ? k * bb : 0);
    double v = 0.0;
    if (INVERT) {
        double *m = bsm + (w * per + (on ? g : 0)) * (bb + b), *f = m + bb;
        if (on)
            for (int t = i; t < bb; t += b) m[op == 3 ? t % b * b + t / b : t] = D[t];
        __syncwarp();
        if (!group_invert(m, f, b, on ? i : b) && on) atomicOr(err, AIR_DEVERR_SINGULAR);
        if (on)
            for (int j = 0; j < b; ++j) v += m[i * b + j] * x[k * b + j];
    } else if (on) {
        for (int j = 0; j < b; ++j) v += D[op == 1 ? j * b + i : i * b + j] * x[k * b + j];
    }
    __syncwarp();
    if (on) y[k * b + i] = v;
}

}  // namespace

int air_csr_transpose_impl(int64_t n, int64_t ncols, int64_t nnz, const int64_t *rp, const int32_t *ci,
                           const double *v, int64_t *rpt, int32_t *cit, double *vt, int *d_err, cudaStream_t s) {
    int32_t *cnt = nullptr;
    AIR_CUDA(cudaMallocAsync(&cnt, (size_t)(ncols > 0 ? ncols : 1) * sizeof(int32_t), s));
    AIR_CUDA(cudaMemsetAsync(cnt, 0, (size_t)(ncols > 0 ? ncols : 1) * sizeof(int32_t), s));
    if (nnz > 0) {
        col_count_kernel<<<air_counted(blocks_for(nnz, 256)), 256, 0, s>>>(nnz, ci, ncols, cnt, d_err);
        AIR_LAUNCH();
    }
    int st = air_exclusive_scan_i32(cnt, rpt, ncols, s);
    if (st == AIR_OK) {
        AIR_CUDA(cudaMemsetAsync(cnt, 0, (size_t)(ncols > 0 ? ncols : 1) * sizeof(int32_t), s));
        scatter_t_kernel<<<air_counted(blocks_for(n, 256)), 256, 0, s>>>(n, rp, ci, v, ncols, rpt, cnt, cit, vt);
        AIR_LAUNCH();
        sort_rows_kernel<<<air_counted(blocks_for(ncols * 32, 256)), 256, 0, s>>>(ncols, rpt, cit, vt);
        AIR_LAUNCH();
    }
    cudaFreeAsync(cnt, s);
    return st;
}

int air_csr_outer_impl(int64_t n, int64_t ncols, const int64_t *rp, const int32_t *ci, const double *u,
                       const double *w, double alpha, double *out, cudaStream_t s) {
    if (n <= 0) return AIR_OK;
    outer_kernel<<<air_counted(blocks_for(n * 32, 256)), 256, 0, s>>>(n, ncols, rp, ci, u, w, alpha, out);
    AIR_LAUNCH();
    return AIR_OK;
}

int air_block_scale_transpose_impl(int64_t n, int b, const double *diag, const int64_t *rpt, const int32_t *cit,
                                   double *vt, int *d_err, cudaStream_t s) {
    const int64_t nblk = n / b;
    if (nblk <= 0) return AIR_OK;
    const size_t smem = (size_t)4 * (1 + 3 * SCALE_CH) * b * b * sizeof(double);
    AIR_CUDA(air_smem_optin(block_scale_t_kernel));
    double *inv = nullptr;
    AIR_CUDA(cudaMallocAsync(&inv, (size_t)(nblk * b * b) * sizeof(double), s));
    invert_transposed_kernel<<<air_counted((unsigned)((nblk + 31) / 32)), 32, b * b * LANE_LD * sizeof(double), s>>>(
        nblk, b, diag, inv, d_err);
    block_scale_t_kernel<<<air_counted((unsigned)((nblk + 3) / 4)), 128, smem, s>>>(nblk, b, diag, inv, rpt, cit, vt,
                                                                                     d_err);
    const cudaError_t e = cudaGetLastError();
    cudaFreeAsync(inv, s);
    AIR_CUDA(e);
    return AIR_OK;
}

int air_block_apply_impl(int64_t nblk, int b, const double *diag, int op, const double *x, double *y, int *d_err,
                         cudaStream_t s) {
    if (nblk <= 0) return AIR_OK;
    const int per = 4 * (32 / b);
    const unsigned groups = (unsigned)((nblk + per - 1) / per);
    if (op < 2)
        block_rows_kernel<false><<<air_counted(groups), 128, 0, s>>>(nblk, b, diag, op, x, y, d_err);
    else
        block_rows_kernel<true><<<air_counted(groups), 128, per * (b * b + b) * sizeof(double), s>>>(nblk, b, diag, op, x,
                                                                                                    y, d_err);
    AIR_LAUNCH();
    return AIR_OK;
}
