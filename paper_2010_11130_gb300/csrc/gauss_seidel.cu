// Forward Gauss-Seidel relaxation, the paper's post-relaxation (Section 4
// settings: forward Gauss-Seidel on the F points, then on all points), in
// ascending point order on every level, as sweeps the relaxation string
// selects with 'f' (F points), 'c' (C points) and 'a' (all points).
//
// A sweep over a point set S updates i in S in ascending order with the
// values already updated: x_i <- x_i + omega (b_i - sum_j a_ij x_j) / a_ii,
// where x_j is new for j < i and old for j >= i.  Rows with no coupling to a
// lower-index row of S depend on nothing; grouping every row by its depth in
// the graph of lower-index couplings inside S gives groups whose rows are
// independent, and processing the groups in depth order reproduces the
// sequential sweep exactly.  The schedule, the rows in depth order, is built
// once at setup by a frontier traversal, one launch per depth.
//
// A sweep is one launch: warps take rows of the schedule in order from a
// ticket counter and wait for the values they need.  A value is its own
// signal: xn starts as a bit pattern no sweep stores wherever the set will
// write, so a row polls x_j itself and needs no flags and no fences.  Only
// earlier rows are waited for, and those were taken by warps that already
// run, so the sweep ends whatever part of its grid is resident and whatever
// else runs beside it; polls are bounded all the same, and a wait that runs out
// is reported by the next solve or air_hierarchy_status.  What bounds it is the
// chain of depth groups: one hop, a store and a poll through the L2 (0.44 us
// between two lanes) and one row's sum, takes 0.9 to 1 us, against 6 us for a
// launch per group.  One lane per entry: with two, four or eight entries per
// lane, polled one after the other, a hop takes 1.1, 1.3 and 2.5 us.  The
// V-cycle with "fa" on 120,150 unknowns (1,500 groups): 1.6 ms (9.3 ms).
#include <type_traits>

#include "air_internal.cuh"

namespace {

constexpr unsigned FULL = 0xffffffffu;

unsigned grid_for(int64_t items, int threads) {
    int64_t b = (items + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > 152 * 32) b = 152 * 32;
    return (unsigned)b;
}

__device__ __forceinline__ bool in_set(const int8_t *cf, int which, int64_t j) {
    return which == 2 || cf[j] == which;
}

// in-degree (lower-index couplings inside the set) and the out-degree counts of the transposed graph
__global__ void gs_degree_kernel(int64_t n, const int64_t *rp, const int32_t *ci, const int8_t *cf, int which,
                                 int32_t *indeg, int32_t *outdeg) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        if (!in_set(cf, which, i)) { indeg[i] = -1; continue; }
        int d = 0;
        for (int64_t k = rp[i]; k < rp[i + 1]; ++k) {
            const int32_t j = ci[k];
            if (j < i && in_set(cf, which, j)) { ++d; atomicAdd(&outdeg[j], 1); }
        }
        indeg[i] = d;
    }
}

__global__ void gs_succ_kernel(int64_t n, const int64_t *rp, const int32_t *ci, const int8_t *cf, int which,
                               const int64_t *optr, int32_t *fill, int32_t *succ) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        if (!in_set(cf, which, i)) continue;
        for (int64_t k = rp[i]; k < rp[i + 1]; ++k) {
            const int32_t j = ci[k];
            if (j < i && in_set(cf, which, j)) succ[optr[j] + atomicAdd(&fill[j], 1)] = (int32_t)i;
        }
    }
}

__global__ void gs_roots_kernel(int64_t n, const int32_t *indeg, int32_t *rows, unsigned long long *tail) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        if (indeg[i] == 0) rows[atomicAdd(tail, 1ull)] = (int32_t)i;
}

// one depth step: successors whose last lower-index coupling was just placed join the next group
__global__ void gs_advance_kernel(int64_t a, int64_t b, const int64_t *optr, const int32_t *succ, int32_t *indeg,
                                  int32_t *rows, unsigned long long *tail) {
    for (int64_t t = a + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < b; t += (int64_t)gridDim.x * blockDim.x) {
        const int32_t i = rows[t];
        for (int64_t k = optr[i]; k < optr[i + 1]; ++k) {
            const int32_t sx = succ[k];
            if (atomicSub(&indeg[sx], 1) == 1) rows[atomicAdd(tail, 1ull)] = sx;
        }
    }
}

// The bit pattern of a value not yet written (a NaN that arithmetic does not
// produce), and polls through the L2.
template <typename T>
struct Slot;
template <>
struct Slot<double> {
    using bits = unsigned long long;
    static constexpr bits PENDING = ~0ull, QNAN = 0x7ff8000000000000ull;
    static __device__ __forceinline__ bits load(const double *p) {
        bits v;
        asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
        return v;
    }
    static __device__ __forceinline__ void store(double *p, bits v) {
        asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
    }
    static __device__ __forceinline__ bits of(double x) { return (bits)__double_as_longlong(x); }
    static __device__ __forceinline__ double value(bits v) { return __longlong_as_double((long long)v); }
};
template <>
struct Slot<float> {
    using bits = unsigned;
    static constexpr bits PENDING = ~0u, QNAN = 0x7fc00000u;
    static __device__ __forceinline__ bits load(const float *p) {
        bits v;
        asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
        return v;
    }
    static __device__ __forceinline__ void store(float *p, bits v) {
        asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
    }
    static __device__ __forceinline__ bits of(float x) { return __float_as_uint(x); }
    static __device__ __forceinline__ float value(bits v) { return __uint_as_float(v); }
};

// what a row stores: x, with the pending pattern (a NaN of the caller's data) replaced by another NaN
template <typename T>
__device__ __forceinline__ typename Slot<T>::bits settled(T x) {
    const typename Slot<T>::bits v = Slot<T>::of(x);
    return v == Slot<T>::PENDING ? Slot<T>::QNAN : v;
}

// xn = pending on the set, x elsewhere; the ticket counter starts at zero
template <typename T>
__global__ void gs_begin_kernel(int64_t n, const int8_t *cf, int which, const T *x, T *xn, unsigned *ticket) {
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t0 == 0) *ticket = 0u;
    for (int64_t i = t0; i < n; i += (int64_t)gridDim.x * blockDim.x)
        xn[i] = Slot<T>::value(in_set(cf, which, i) ? Slot<T>::PENDING : settled(x[i]));
}

// One warp per row, one lane per entry: rows order[c K] .. order[c K + K - 1] of ticket c.  The entries' products are
// summed in FP32 as `vl` lanes with every vl-th entry each would sum them (the order of the sets' storage), in FP64 by
// a tree over the warp (a dependent DFMA takes 64 cycles here, an FP32 one 7).
template <typename T>
__global__ void __launch_bounds__(128) gs_sweep_kernel(int64_t m, int K, int vl, const int32_t *__restrict__ order,
                                                       const int64_t *__restrict__ rp, const int32_t *__restrict__ ci,
                                                       const T *__restrict__ v, const T *__restrict__ xo, T *xn,
                                                       const T *__restrict__ b, const T *__restrict__ dinv, T omega,
                                                       unsigned *ticket, int polls_cap, int *err) {
    using S = Slot<T>;
    const int lane = threadIdx.x & 31;
    unsigned c = 0;
    if (lane == 0) c = atomicAdd(ticket, 1u);
    c = __shfl_sync(FULL, c, 0);
    while ((int64_t)c * K < m) {
        unsigned next = 0;                // taken early: its latency passes behind these rows
        if (lane == 0) next = atomicAdd(ticket, 1u);
        const int64_t end = (int64_t)(c + 1) * K < m ? (int64_t)(c + 1) * K : m;
        for (int64_t t = (int64_t)c * K; t < end; ++t) {
            const int64_t i = order[t], rs = rp[i], re = rp[i + 1];
            const T xi = xo[i], bi = b[i], di = dinv[i];
            T acc = 0;
            for (int64_t k0 = rs; k0 < re; k0 += 32) {
                const bool on = k0 + lane < re;
                const int32_t j = on ? ci[k0 + lane] : INT32_MAX;
                const T a = on ? v[k0 + lane] : (T)0;
                T x = 0;
                if (j < i) {
                    typename S::bits w = S::load(xn + j);
                    int polls = 0;
                    while (w == S::PENDING && ++polls < polls_cap) w = S::load(xn + j);
                    if (w == S::PENDING) {
                        atomicOr(err, AIR_DEVERR_RS_CAP);
                        w = S::QNAN;
                    }
                    x = S::value(w);
                } else if (on) {
                    x = xo[j];
                }
                __syncwarp();
                if (std::is_same<T, double>::value) {
                    acc += a * x;
                } else {
                    for (int q = lane % vl; q < 32; q += vl) {
                        const T aq = __shfl_sync(FULL, a, q), xq = __shfl_sync(FULL, x, q);
                        acc += aq * xq;
                    }
                }
            }
            const int width = std::is_same<T, double>::value ? 32 : vl;
            for (int o = width / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(FULL, acc, o);
            if (lane == 0) S::store(xn + i, settled<T>(xi + omega * (bi - acc) * di));
        }
        c = __shfl_sync(FULL, next, 0);
    }
}

// Lanes whose partial sums an FP32 row's sum stands for: every lane at most eight entries of the mean row.
int lanes_for(const AirLevel &L) {
    const double avg = L.n > 0 ? (double)L.nnz / (double)L.n : 1.0;
    int vl = 1;
    while (vl < 32 && avg / vl > 8.0) vl *= 2;
    return vl;
}

int build_one(AirLevel &L, int which, cudaStream_t s) {
    AirLevel::GsSchedule &G = L.gs[which];
    const int64_t n = L.n;
    int32_t *indeg = nullptr, *outdeg = nullptr, *fill = nullptr, *succ = nullptr;
    int64_t *optr = nullptr;
    unsigned long long *tail = nullptr;
    AIR_CUDA(cudaMallocAsync(&indeg, (size_t)n * sizeof(int32_t), s));
    AIR_CUDA(cudaMallocAsync(&outdeg, (size_t)n * sizeof(int32_t), s));
    AIR_CUDA(cudaMemsetAsync(outdeg, 0, (size_t)n * sizeof(int32_t), s));
    gs_degree_kernel<<<air_counted(grid_for(n, 256)), 256, 0, s>>>(n, L.rp, L.ci, L.cf, which, indeg, outdeg);
    AIR_LAUNCH();
    AIR_CUDA(cudaMallocAsync(&optr, (size_t)(n + 1) * sizeof(int64_t), s));
    AIR_TRY(air_exclusive_scan_i32(outdeg, optr, n, s));
    int64_t ne = 0;
    AIR_CUDA(cudaMemcpyAsync(&ne, optr + n, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    AIR_CUDA(cudaStreamSynchronize(s));
    AIR_CUDA(cudaMallocAsync(&succ, (size_t)(ne > 0 ? ne : 1) * sizeof(int32_t), s));
    AIR_CUDA(cudaMallocAsync(&fill, (size_t)n * sizeof(int32_t), s));
    AIR_CUDA(cudaMemsetAsync(fill, 0, (size_t)n * sizeof(int32_t), s));
    gs_succ_kernel<<<air_counted(grid_for(n, 256)), 256, 0, s>>>(n, L.rp, L.ci, L.cf, which, optr, fill, succ);
    AIR_LAUNCH();
    const int64_t m = which == 2 ? n : (which == 1 ? L.nc : L.nf);
    int32_t *order = nullptr;
    AIR_CUDA(air_dmalloc((void **)&order, (size_t)(m > 0 ? m : 1) * sizeof(int32_t)));
    AIR_CUDA(cudaMallocAsync(&tail, sizeof(unsigned long long), s));
    AIR_CUDA(cudaMemsetAsync(tail, 0, sizeof(unsigned long long), s));
    gs_roots_kernel<<<air_counted(grid_for(n, 256)), 256, 0, s>>>(n, indeg, order, tail);
    AIR_LAUNCH();
    int32_t depth = 0;
    unsigned long long h = 0;
    AIR_CUDA(cudaMemcpyAsync(&h, tail, sizeof(h), cudaMemcpyDeviceToHost, s));
    AIR_CUDA(cudaStreamSynchronize(s));
    int64_t a = 0, b = (int64_t)h;
    while (b > a) {
        if (++depth > m) break;                      // cannot happen: the graph is acyclic
        gs_advance_kernel<<<air_counted(grid_for(b - a, 256)), 256, 0, s>>>(a, b, optr, succ, indeg, order, tail);
        AIR_LAUNCH();
        AIR_CUDA(cudaMemcpyAsync(&h, tail, sizeof(h), cudaMemcpyDeviceToHost, s));
        AIR_CUDA(cudaStreamSynchronize(s));
        a = b;
        b = (int64_t)h;
    }
    cudaFreeAsync(indeg, s);
    cudaFreeAsync(outdeg, s);
    cudaFreeAsync(fill, s);
    cudaFreeAsync(succ, s);
    cudaFreeAsync(optr, s);
    cudaFreeAsync(tail, s);
    if (b != m) {                                     // every row of the set must be placed
        air_dfree(order);
        return AIR_ERR_CUDA;
    }
    G.m = m;
    G.depth = depth;
    G.dev_rows = order;
    AIR_CUDA(air_dmalloc((void **)&G.ticket, sizeof(unsigned)));
    return AIR_OK;
}

__global__ void d2f_values_kernel(int64_t n, const double *in, float *out) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = (float)in[i];
}

}  // namespace

int air_gs_build(air_hierarchy *H, cudaStream_t s) {
    bool need[3] = {false, false, false};
    for (const char *c = H->opt.relax; *c; ++c) {
        if (*c == 'f') need[0] = true;
        if (*c == 'c') need[1] = true;
        if (*c == 'a') need[2] = true;
    }
    if (!need[0] && !need[1] && !need[2]) return AIR_OK;
    H->gs = true;
    for (int q = 0; q + 1 < H->nlev; ++q) {
        AirLevel &L = H->lev[q];
        for (int w = 0; w < 3; ++w)
            if (need[w]) AIR_TRY(build_one(L, w, s));
        if (H->opt.precision == AIR_PREC_F32) {
            AIR_CUDA(air_dmalloc((void **)&L.v32, (size_t)(L.nnz > 0 ? L.nnz : 1) * sizeof(float)));
            d2f_values_kernel<<<air_counted(grid_for(L.nnz, 256)), 256, 0, s>>>(L.nnz, L.v, L.v32);
            AIR_LAUNCH();
        }
    }
    return AIR_OK;
}

void air_gs_free(AirLevel &L) {
    for (auto &G : L.gs) {
        air_dfree(G.dev_rows);
        air_dfree(G.ticket);
        G = AirLevel::GsSchedule();
    }
    air_dfree(L.v32);
    L.v32 = nullptr;
}

int air_gs_fetch(const air_hierarchy *H, int *flags, cudaStream_t s) {
    if (!H->gs) return AIR_OK;
    AIR_CUDA(cudaMemcpyAsync(flags, H->d_err, sizeof(int), cudaMemcpyDeviceToHost, s));
    return AIR_OK;
}

int air_gs_take(const air_hierarchy *H, const int *flags, cudaStream_t s) {
    if (!H->gs || !(*flags & AIR_DEVERR_RS_CAP)) return AIR_OK;
    AIR_CUDA(cudaMemsetAsync(H->d_err, 0, sizeof(int), s));
    AIR_CUDA(cudaStreamSynchronize(s));
    return AIR_ERR_DEVICE_TIMEOUT;
}

template <typename T>
int air_gs_sweep(const AirLevel &L, int which, T omega, const T *b, const T *x, T *xn, int polls, int *err,
                 cudaStream_t s) {
    const AirLevel::GsSchedule &G = L.gs[which];
    const bool f64 = std::is_same<T, double>::value;
    const T *dinv = f64 ? (const T *)L.dinv : (const T *)L.dinv32;
    const T *v = f64 ? (const T *)L.v : (const T *)L.v32;
    gs_begin_kernel<T><<<air_counted(grid_for(L.n, 256)), 256, 0, s>>>(L.n, L.cf, which, x, xn, G.ticket);
    if (G.m > 0) {
        // Eight mean group widths of warps, so that the rows of the groups behind the one that is ready are loaded
        // while they wait (four: 6% slower, one: 60%), between 16 blocks and eight blocks per SM.  Where even one
        // group is wider than that, a ticket stands for several rows, so that the counter does not bound the sweep.
        const double width = (double)G.m / (double)G.depth, most = 152.0 * 8.0 * 4.0;
        double warps = 8.0 * width < 64.0 ? 64.0 : (8.0 * width > most ? most : 8.0 * width);
        if (warps > (double)G.m) warps = (double)G.m;
        const int K = width > most ? (width > 8.0 * most ? 8 : (int)(width / most)) : 1;
        gs_sweep_kernel<T><<<air_counted((unsigned)((warps + 3.0) / 4.0)), 128, 0, s>>>(
            G.m, K, lanes_for(L), G.dev_rows, L.rp, L.ci, v, x, xn, b, dinv, omega, G.ticket, polls, err);
    }
    AIR_LAUNCH();
    return AIR_OK;
}

template int air_gs_sweep<double>(const AirLevel &, int, double, const double *, const double *, double *, int,
                                  int *, cudaStream_t);
template int air_gs_sweep<float>(const AirLevel &, int, float, const float *, const float *, float *, int, int *,
                                 cudaStream_t);
