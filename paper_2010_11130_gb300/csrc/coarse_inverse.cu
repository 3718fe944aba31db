// Explicit inverse of the coarsest operator (arXiv:2010.11130, Section 3: the
// correction's coarse solve; the V-cycle applies it as one matrix-vector
// product): blocked in-place Gauss-Jordan with partial pivoting (ties ->
// smallest row), PB columns at a time.
//
//  - panel_kernel, one cluster: the PB columns of a panel are eliminated with
//    one row per thread in registers.  A step needs one cluster barrier: every
//    block pushes its best pivot candidate, that row divided by its pivot and,
//    from its owner, row k to all blocks, and every thread picks the winner for
//    itself.  One more barrier, behind the loads of the rows, comes before the
//    first push.  The rows' multipliers are kept by the row they belong to.
//  - pivot_rows_kernel: the panel's rows of every other column, step by step.
//  - update_kernel, all SMs: the panel's steps on every other entry, in order,
//    reading the old matrix through the panel's row swaps and writing the other
//    buffer.
//  - the row swaps are undone on the columns at the end.
// Every entry goes through the operations of the unblocked elimination in
// their order (a / pivot, then fma(-f, a_kj, a_ij) for k = 0, 1, ...), so the
// inverse, and the FP32 copy of it, are the same bits.
//
// What bounds it: n^3 FP64 multiply-adds in the updates (1.6 ms for n = 991 at
// two per SM and clock) and the chain of n pivot steps (about 2 us each: a
// division, 16 dependent-rate FP64 instructions per row, one barrier).
// n = 991: 6.0 ms for the inverse (15 to 25 ms with two grid barriers and a full
// pass over [A | I] per column).
#include <cooperative_groups.h>
#include <math.h>

#include "air_internal.cuh"
#include "lane_dense.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int PB = 16;            // panel columns
constexpr int CL = 8;             // blocks of the panel's cluster
constexpr int PT = 512;           // most threads of a panel block
constexpr int TILE = 32;          // update tile

unsigned grid_for(int64_t items, int threads, int64_t cap = 152 * 16) {
    int64_t b = (items + threads - 1) / threads;
    return (unsigned)(b < 1 ? 1 : (b > cap ? cap : b));
}

__global__ void dense_scatter_kernel(int64_t n, const int64_t *rp, const int32_t *ci, const double *v, double *M,
                                     unsigned long long *amax) {
    unsigned long long top = 0ull;    // magnitudes as integers: their order is the same
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        for (int64_t k = rp[i]; k < rp[i + 1]; ++k) {
            M[i * n + ci[k]] = v[k];
            const unsigned long long m = magnitude_key(v[k]);
            top = m > top ? m : top;
        }
    if (top > 1ull) atomicMax(amax, top - 1ull);
}

struct PanelArgs {
    int64_t n, k0, chunk;         // order, first column of the panel, rows per block
    int nb;                       // columns of the panel
    double *M;                    // n x n, old matrix
    double *T;                    // n x PB: the panel's columns after its steps
    double *F;                    // n x PB: multipliers of every row of the old matrix, by that row
    double *piv_val;              // PB pivots
    int32_t *src;                 // row of the old matrix at every position after the panel's swaps
    int32_t *piv;                 // pivot position of every column
    const unsigned long long *amax;
    int *err;
};

struct Candidate {                // a pivot row offered by one block
    double s[PB];                 // the row over its pivot; the reciprocal in the pivot's column
    double pivot;
    unsigned long long key;
    long long row, id;            // position, and row of the old matrix there
};
constexpr int CW = sizeof(Candidate) / 8;

// REG: at most PT rows per block, one per thread, in registers; otherwise the threads loop over their rows in T.
template <bool REG>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(PT) panel_kernel(PanelArgs g) {
    __shared__ Candidate cand[2][CL], mine;
    __shared__ double krow[2][PB + 1], mykrow[PB + 1];          // row k and, last, its row of the old matrix
    __shared__ unsigned long long wkey[PT / 32];
    __shared__ long long wrow[PT / 32];
    cg::cluster_group cluster = cg::this_cluster();
    const int tid = threadIdx.x, lane = tid & 31, nw = blockDim.x >> 5, rank = (int)cluster.block_rank();
    if (*(volatile int *)g.err & AIR_DEVERR_SINGULAR) return;         // an earlier panel; the same for all blocks
    // A block's shared memory may be written by the others once it runs: all arrive here and wait below, before the
    // first remote write.
    cluster.barrier_arrive();
    const int64_t lo = rank * g.chunk, hi = lo + g.chunk < g.n ? lo + g.chunk : g.n;
    const double tol = 1e-14 * __longlong_as_double((long long)*g.amax);
    double a[PB];
    for (int64_t r = lo + tid; r < hi; r += blockDim.x) {
        g.src[r] = (int32_t)r;
#pragma unroll
        for (int c = 0; c < PB; ++c) {
            const double x = c < g.nb ? g.M[r * g.n + g.k0 + c] : 0.0;
            if (REG) a[c] = x;
            else g.T[r * PB + c] = x;
        }
    }
    int32_t id = (int32_t)(lo + tid);                  // REG: the row of the old matrix the thread holds
    cluster.barrier_wait();
    for (int c = 0; c < g.nb; ++c) {
        const int64_t k = g.k0 + c;
        const int par = c & 1;
        unsigned long long best = 0ull;
        long long br = g.n;
        for (int64_t r = lo + tid; r < hi; r += blockDim.x) {
            if (r < k) continue;
            double x = 0.0;
            if (REG) {
#pragma unroll
                for (int q = 0; q < PB; ++q) x = q == c ? a[q] : x;
            } else {
                x = g.T[r * PB + c];
            }
            const unsigned long long key = magnitude_key(x);
            if (key > best) { best = key; br = r; }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long ok = __shfl_xor_sync(FULL, best, o);
            const long long orow = __shfl_xor_sync(FULL, br, o);
            if (ok > best || (ok == best && orow < br)) { best = ok; br = orow; }
        }
        if (lane == 0) { wkey[tid >> 5] = best; wrow[tid >> 5] = br; }
        __syncthreads();
        for (int w = 0; w < nw; ++w)
            if (wkey[w] > best || (wkey[w] == best && wrow[w] < br)) { best = wkey[w]; br = wrow[w]; }
        if (tid == 0) { mine.key = best; mine.row = br; }
        for (int64_t r = lo + tid; r < hi; r += blockDim.x) {
            if (r == br) {
                mine.id = REG ? id : g.src[r];
#pragma unroll
                for (int q = 0; q < PB; ++q) {
                    const double x = REG ? a[q] : g.T[r * PB + q];
                    mine.s[q] = x;
                    if (q == c) mine.pivot = x;
                }
            }
            if (r == k) {
                mykrow[PB] = __longlong_as_double((long long)(REG ? id : g.src[r]));
#pragma unroll
                for (int q = 0; q < PB; ++q) mykrow[q] = REG ? a[q] : g.T[r * PB + q];
            }
        }
        __syncthreads();
        if (tid < PB && best > 1ull) mine.s[tid] = (tid == c ? 1.0 : mine.s[tid]) / mine.pivot;
        __syncthreads();
        const bool has_k = lo <= k && k < hi;
        for (int t = tid; t < CL * CW; t += blockDim.x)
            ((unsigned long long *)cluster.map_shared_rank(&cand[par][rank], t / CW))[t % CW] =
                ((const unsigned long long *)&mine)[t % CW];
        if (has_k)
            for (int t = tid; t < CL * (PB + 1); t += blockDim.x)
                cluster.map_shared_rank(&krow[par][0], t / (PB + 1))[t % (PB + 1)] = mykrow[t % (PB + 1)];
        cluster.sync();
        int win = 0;
#pragma unroll
        for (int q = 1; q < CL; ++q)
            if (cand[par][q].key > cand[par][win].key ||
                (cand[par][q].key == cand[par][win].key && cand[par][q].row < cand[par][win].row))
                win = q;
        const Candidate &P = cand[par][win];
        const int64_t p = P.row;
        // nothing above the tolerance: every thread of every block sees it and leaves (the last barrier is behind them)
        if (P.key <= 1ull || !(fabs(P.pivot) > tol)) {
            if (rank == 0 && tid == 0) atomicOr(g.err, AIR_DEVERR_SINGULAR);
            return;
        }
        if (rank == 0 && tid == 0) {
            g.piv[k] = (int32_t)p;
            g.piv_val[c] = P.pivot;
        }
        for (int64_t r = lo + tid; r < hi; r += blockDim.x) {
            // position k takes the divided pivot row (as a zero row minus -1 times it), position p the row that was at k
            int32_t row = REG ? id : g.src[r];
            double v[PB], f = 0.0;
#pragma unroll
            for (int q = 0; q < PB; ++q) {
                v[q] = REG ? a[q] : g.T[r * PB + q];
                if (r == p) v[q] = krow[par][q];
                f = q == c ? v[q] : f;
                if (r == k || q == c) v[q] = 0.0;
            }
            if (r == p) row = (int32_t)__double_as_longlong(krow[par][PB]);
            if (r == k) {
                row = (int32_t)P.id;
                f = -1.0;
            }
            if (REG) id = row;
            else g.src[r] = row;
            g.F[(int64_t)row * PB + c] = f;
#pragma unroll
            for (int q = 0; q < PB; ++q) {
                const double x = fma(-f, P.s[q], v[q]);
                if (REG) a[q] = x;
                else g.T[r * PB + q] = x;
            }
        }
        if (!REG) __syncthreads();
    }
    if (REG && lo + tid < hi) {
        g.src[lo + tid] = id;
#pragma unroll
        for (int q = 0; q < PB; ++q) g.T[(lo + tid) * PB + q] = a[q];
    }
}

// S(c, j): row k0 + c of column j right after its own step of the panel, one thread per column.
__global__ void __launch_bounds__(128) pivot_rows_kernel(int64_t n, int64_t k0, int nb, const double *__restrict__ A,
                                                         const double *__restrict__ F, const double *piv_val,
                                                         const int32_t *__restrict__ src, double *__restrict__ S,
                                                         const int *err) {
    __shared__ double sF[PB][PB];
    __shared__ double sd[PB];
    if (*err & AIR_DEVERR_SINGULAR) return;
    for (int t = threadIdx.x; t < PB * PB; t += blockDim.x)
        sF[t / PB][t % PB] = t / PB < nb && t % PB < nb ? F[(int64_t)src[k0 + t / PB] * PB + t % PB] : 0.0;
    if (threadIdx.x < PB) sd[threadIdx.x] = (int)threadIdx.x < nb ? piv_val[threadIdx.x] : 1.0;
    __syncthreads();
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    double w[PB];
#pragma unroll
    for (int c = 0; c < PB; ++c) w[c] = c < nb ? A[(int64_t)src[k0 + c] * n + j] : 0.0;
#pragma unroll
    for (int c = 0; c < PB; ++c) {
        w[c] = w[c] / sd[c];
#pragma unroll
        for (int q = c + 1; q < PB; ++q) w[q] = fma(-sF[q][c], w[c], w[q]);
    }
#pragma unroll
    for (int c = 0; c < PB; ++c) S[c * n + j] = w[c];
}

// B(i, j) = T(i, j - k0) in the panel's columns; elsewhere A(src i, j), or S(i - k0, j) in the panel's rows, after the
// steps of the panel (in its rows: the steps after their own).  One 32 x 32 tile per block.
__global__ void __launch_bounds__(256) update_kernel(int64_t n, int64_t k0, int nb, const double *__restrict__ A,
                                                     const double *__restrict__ T, const double *__restrict__ F,
                                                     const double *__restrict__ S, const int32_t *__restrict__ src,
                                                     double *__restrict__ B, const int *err) {
    __shared__ double sF[TILE][PB + 1], sS[PB][TILE];
    if (*err & AIR_DEVERR_SINGULAR) return;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int64_t i0 = (int64_t)blockIdx.y * TILE, j = (int64_t)blockIdx.x * TILE + tx;
    for (int t = threadIdx.x; t < TILE * PB; t += 256) {
        const int64_t i = i0 + t / PB;
        const int c = t % PB;
        const bool on = i < n && c < nb && (i < k0 || i >= k0 + nb || c > i - k0);
        sF[t / PB][c] = on ? F[(int64_t)src[i] * PB + c] : 0.0;
    }
    for (int c = ty; c < PB; c += 8) sS[c][tx] = c < nb && j < n ? S[c * n + j] : 0.0;
    double acc[TILE / 8];
#pragma unroll
    for (int u = 0; u < TILE / 8; ++u) {
        const int64_t i = i0 + ty + 8 * u;
        acc[u] = i >= n || j >= n ? 0.0 : (i < k0 || i >= k0 + nb ? A[(int64_t)src[i] * n + j] : S[(i - k0) * n + j]);
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < PB; ++c)
#pragma unroll
        for (int u = 0; u < TILE / 8; ++u) acc[u] = fma(-sF[ty + 8 * u][c], sS[c][tx], acc[u]);
    if (j >= n) return;
    const bool panel = j >= k0 && j < k0 + nb;
#pragma unroll
    for (int u = 0; u < TILE / 8; ++u) {
        const int64_t i = i0 + ty + 8 * u;
        if (i < n) B[i * n + j] = panel ? T[i * PB + j - k0] : acc[u];
    }
}

// col[j]: the column of the eliminated matrix that is column j of the inverse (the row swaps undone, last first), in
// shared memory when it holds the n integers
__global__ void column_order_kernel(int64_t n, const int32_t *piv, int32_t *col, bool shared, const int *err) {
    extern __shared__ int32_t scol[];
    int32_t *order = shared ? scol : col;
    if (*err & AIR_DEVERR_SINGULAR) return;
    for (int64_t t = threadIdx.x; t < n; t += blockDim.x) order[t] = (int32_t)t;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int64_t k = n - 1; k >= 0; --k) {
            const int32_t p = piv[k], x = order[k];
            order[k] = order[p];
            order[p] = x;
        }
    __syncthreads();
    for (int64_t t = threadIdx.x; t < n; t += blockDim.x) col[t] = order[t];
}

__global__ void dense_extract_kernel(int64_t n, const double *M, const int32_t *col, double *inv, const int *err) {
    if (*err & AIR_DEVERR_SINGULAR) return;
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n * n; s += (int64_t)gridDim.x * blockDim.x)
        inv[s] = M[s / n * n + col[s % n]];
}

}  // namespace

int air_coarse_inverse(int64_t n, const int64_t *rp, const int32_t *ci, const double *v, double *inv, int *d_err,
                       cudaStream_t s) {
    const size_t order_bytes = (size_t)n * sizeof(int32_t);
    const bool shared = order_bytes <= AIR_SMEM_OPTIN;
    AIR_CUDA(air_smem_optin(column_order_kernel));
    // two matrices, the panel's columns, multipliers and rows, its pivots, then the integers
    double *work = nullptr;
    AIR_CUDA(cudaMallocAsync((void **)&work, (size_t)(2 * n * n + 3 * PB * n + PB + 1) * sizeof(double) + 3 * order_bytes, s));
    double *A = work, *B = A + n * n, *T = B + n * n, *F = T + PB * n, *S = F + PB * n, *pv = S + PB * n;
    unsigned long long *amax = (unsigned long long *)(pv + PB);
    int32_t *src = (int32_t *)(amax + 1), *piv = src + n, *col = piv + n;
    cudaError_t e = cudaMemsetAsync(A, 0, (size_t)(n * n) * sizeof(double), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(amax, 0, sizeof(*amax), s);
    dense_scatter_kernel<<<air_counted(grid_for(n, 128)), 128, 0, s>>>(n, rp, ci, v, A, amax);
    const int64_t chunk = (n + CL - 1) / CL, width = chunk < PT ? (chunk + 31) / 32 * 32 : PT;
    const unsigned threads = (unsigned)(width < 128 ? 128 : width);
    const unsigned tiles = (unsigned)((n + TILE - 1) / TILE);
    for (int64_t k0 = 0; k0 < n; k0 += PB) {
        PanelArgs g{n, k0, chunk, n - k0 < PB ? (int)(n - k0) : PB, A, T, F, pv, src, piv, amax, d_err};
        if (chunk <= (int64_t)threads) panel_kernel<true><<<air_counted(CL), threads, 0, s>>>(g);
        else panel_kernel<false><<<air_counted(CL), threads, 0, s>>>(g);
        pivot_rows_kernel<<<air_counted((unsigned)((n + 31) / 32)), 32, 0, s>>>(n, k0, g.nb, A, F, pv, src, S, d_err);
        update_kernel<<<air_counted(dim3(tiles, tiles)), 256, 0, s>>>(n, k0, g.nb, A, T, F, S, src, B, d_err);
        double *t = A;
        A = B;
        B = t;
    }
    column_order_kernel<<<air_counted(1), 256, shared ? order_bytes : 0, s>>>(n, piv, col, shared, d_err);
    dense_extract_kernel<<<air_counted(grid_for(n * n, 256)), 256, 0, s>>>(n, A, col, inv, d_err);
    if (e == cudaSuccess) e = cudaGetLastError();
    cudaFreeAsync(work, s);
    AIR_CUDA(e);
    return AIR_OK;
}
