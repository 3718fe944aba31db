// Falgout-style C/F splitting (the coarsening named in the paper's Section 4
// settings, whose details the paper leaves to its library): the points are cut
// into consecutive index blocks of `block` points; the first pass of
// Ruge-Stueben runs in every block at once on the strength graph restricted to
// the block, one warp per block with the block's measures and graph in shared
// memory;
// then the interface points that ended F with strong connections but no
// strong C point are fixed by rounds of a parallel independent set.
//
// Local pass (the single-warp first pass of first_pass.cu, restricted): the
// measure of i is the number of points of its block that depend strongly on
// it; a point with no strong connection inside its block starts F.  Pick the
// undecided point of largest measure, ties to the smallest index; it becomes
// C, its undecided strong dependants in the block become F, every undecided
// point of the block in S_j of a new F point j gains one, every undecided
// point of the block in S_i loses one; stop when the largest measure is 0 (the
// rest become F).  The maximum is found through upper bounds per 32 points that
// increments raise and searches repair when they meet a stale one; the largest
// bound and its first group come out of one maximum over (bound, group) keys.
// What bounds it is the chain of picks of one block (a block of 8192 points has
// 2,000 to 3,600; blocks run side by side): a pick is a dozen dependent accesses,
// in shared memory 30 cycles each, in the L2 300 to 600.  The block's graph, 16-bit
// local indices both ways, is therefore gathered into shared memory first, and the
// strong connections of up to sixteen new F points are raised together.  All levels
// at 2.3 M unknowns: 13.5 ms (40.8 ms with the graph in global memory and one F point
// after the other, 17.4 ms with two levels of bounds and four F points at a time).
//
// Interface rounds: U = F points with S_i non-empty, no C point in S_i and a
// strong connection (either way) to another block.  Weight
// w_i = |S^T_i| + frac(i), frac from the SplitMix64 hash of i (Steele, Lea and
// Flood, 2014).  A point of U whose weight beats every point of U in S_i and
// S^T_i (ties -> smaller index) becomes C; points of U with a C point in S_i
// leave U; repeat until U is empty.
#include <type_traits>

#include "air_internal.cuh"

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int LT = 1024;             // threads per block of points: all gather its graph, one warp picks
constexpr int NEWF_CAP = 1024;       // new F points of one pick
constexpr int LAM_F = -1, LAM_C = -2;
constexpr int8_t CF_F = 0, CF_C = 1;

__device__ __forceinline__ unsigned lanemask_lt() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

unsigned grid_for(int64_t items, int threads) {
    int64_t b = (items + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > 152 * 32) b = 152 * 32;
    return (unsigned)b;
}

// Shared memory of one block of points: lam[block], g1[block / 32], newF[NEWF_CAP] (int32), then 16
// bits each: row starts of S and of S^T (block + 1, padded to even), their entries (cap each).
struct LocalGraph {
    int64_t lo;                       // first point and number of points
    int m;
    const int64_t *srp, *strp;        // the whole graph, for blocks whose own part does not fit
    const int32_t *sci, *stci;
    const uint16_t *sp, *tp, *se, *te;
};

// Rows of S (T = false) or S^T of a local point, restricted to the block: entry numbers first .. last, at(e) the local
// neighbour or -1 outside the block.
template <bool SMEM, bool T>
struct Row {
    using Entry = typename std::conditional<SMEM, int, int64_t>::type;
    Entry first, last;
    __device__ __forceinline__ Row(const LocalGraph &g, int j) {
        if (SMEM) {
            const uint16_t *p = T ? g.tp : g.sp;
            first = p[j];
            last = p[j + 1];
        } else {
            const int64_t *p = T ? g.strp : g.srp;
            first = p[g.lo + j];
            last = p[g.lo + j + 1];
        }
    }
    __device__ __forceinline__ int at(const LocalGraph &g, Entry e) const {
        if (SMEM) return (T ? g.te : g.se)[e];
        return local(g, (T ? g.stci : g.sci)[e]);
    }
    static __device__ __forceinline__ int local(const LocalGraph &g, int32_t i) {
        const int64_t k = i - g.lo;
        return k >= 0 && k < g.m ? (int)k : -1;
    }
};

// One more for the undecided points in the rows of S listed in newF: eight lanes per row, 4 R rows in flight.
template <bool SMEM, int R>
__device__ __forceinline__ void raise_rows(const LocalGraph &g, int nf, const int32_t *newF, int32_t *lam, int32_t *g1) {
    const int lane = threadIdx.x & 31;
    for (int q0 = lane >> 3; q0 < nf; q0 += 4 * R) {
        typename Row<SMEM, false>::Entry first[R], last[R];
        bool more = false;
#pragma unroll
        for (int u = 0; u < R; ++u) {
            first[u] = last[u] = 0;
            if (q0 + 4 * u < nf) {
                const int32_t f = newF[q0 + 4 * u];
                if (SMEM) {
                    first[u] = (unsigned)f & 0xffffu;
                    last[u] = (unsigned)f >> 16;
                } else {
                    const Row<false, false> r(g, f);
                    first[u] = r.first;
                    last[u] = r.last;
                }
            }
            first[u] += lane & 7;
            more |= first[u] < last[u];
        }
        while (more) {
            int k[R];
            bool up[R];
            more = false;
#pragma unroll
            for (int u = 0; u < R; ++u) {
                k[u] = first[u] < last[u] ? (SMEM ? (int)g.se[first[u]] : Row<false, false>::local(g, g.sci[first[u]])) : -1;
                first[u] += 8;
                more |= first[u] < last[u];
            }
#pragma unroll
            for (int u = 0; u < R; ++u) up[u] = k[u] >= 0 && lam[k[u]] >= 0;
#pragma unroll
            for (int u = 0; u < R; ++u)
                if (up[u]) {
                    const int nv = atomicAdd(&lam[k[u]], 1) + 1;
                    atomicMax(&g1[k[u] >> 5], nv);
                }
        }
    }
}

// The picks of one block, by one warp.
template <bool SMEM>
__device__ void local_picks(const LocalGraph &g, int ng1, int32_t *lam, int32_t *g1, int32_t *newF, int *err) {
    const int lane = threadIdx.x & 31;
    const int64_t cap = 64 * (int64_t)g.m + 1024;  // picks plus repairs of stale bounds (a safety net)
    for (int64_t step = 0;; ++step) {
        if (step > cap) {
            if (lane == 0) atomicOr(err, AIR_DEVERR_RS_CAP);
            break;
        }
        // the largest bound of a 32-point group and the first group that has it, in one maximum: at most 256 groups
        int key = INT32_MIN;
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (32 * u < ng1) {
                const int q = lane + 32 * u;
                key = max(key, g1[q] * 256 + (255 - q));
            }
        key = __reduce_max_sync(FULL, key);
        const int top = key >> 8, q1 = 255 - (key & 255);
        if (top < 1) break;
        const int lv = lam[q1 * 32 + lane];
        const unsigned bal0 = __ballot_sync(FULL, lv == top);
        if (!bal0) {                                   // stale group bound: repair it
            const int mx = __reduce_max_sync(FULL, lv);
            if (lane == 0) g1[q1] = mx;
            __syncwarp();
            continue;
        }
        const int picked = __ffs(bal0) - 1, i = q1 * 32 + picked;
        const Row<SMEM, true> dep(g, i);
        const Row<SMEM, false> own(g, i);
        // i leaves its group: the exact bound now costs less than meeting a stale one later
        const int m1 = __reduce_max_sync(FULL, lane == picked ? LAM_C : lv);
        // undecided strong dependants of i in the block become F; in shared memory newF keeps their row of S (first
        // entry and, from bit 16, the one past the last: below 2^16), loaded beside the measure
        const int k_own = own.first + lane < own.last ? own.at(g, own.first + lane) : -1;
        int nf = 0;
        for (auto a0 = dep.first; a0 < dep.last; a0 += 32) {
            const int j = a0 + lane < dep.last ? dep.at(g, a0 + lane) : -1;
            const int row = SMEM && j >= 0 ? (int)((unsigned)g.sp[j] | (unsigned)g.sp[j + 1] << 16) : j;
            const bool f = j >= 0 && lam[j] >= 0;
            const unsigned bal = __ballot_sync(FULL, f);
            if (f) {
                const int p = nf + __popc(bal & lanemask_lt());
                if (p < NEWF_CAP) newF[p] = row;
                lam[j] = LAM_F;
            }
            nf += __popc(bal);
        }
        if (nf > NEWF_CAP) {
            if (lane == 0) atomicOr(err, AIR_DEVERR_CAP);
            break;
        }
        if (lane == 0) {
            lam[i] = LAM_C;
            g1[q1] = m1;
        }
        __syncwarp();
        // every undecided point of the block in S_i loses one (bounds stay upper bounds, also beside the gains)
        if (k_own >= 0 && lam[k_own] >= 0) atomicSub(&lam[k_own], 1);
        for (auto a = own.first + 32 + lane; a < own.last; a += 32) {
            const int k = own.at(g, a);
            if (k >= 0 && lam[k] >= 0) atomicSub(&lam[k], 1);
        }
        // every undecided point of the block in S_j of a new F point j gains one: eight lanes per j
        if (!SMEM || nf <= 4) raise_rows<SMEM, 1>(g, nf, newF, lam, g1);
        else if (nf <= 8) raise_rows<SMEM, 2>(g, nf, newF, lam, g1);
        else raise_rows<SMEM, 4>(g, nf, newF, lam, g1);
        __syncwarp();
    }
    __syncwarp();
}

__global__ void __launch_bounds__(LT) local_pass_kernel(int64_t n, int64_t block, int cap, const int64_t *srp,
                                                        const int32_t *sci, const int64_t *strp, const int32_t *stci,
                                                        int8_t *cf, int *err) {
    extern __shared__ int32_t fsm[];
    __shared__ int sum[2][LT / 32];
    const int tid = threadIdx.x, lane = tid & 31;
    const int64_t lo = blockIdx.x * block, hi = lo + block < n ? lo + block : n;
    const int m = (int)(hi - lo), ng1 = (int)(block / 32), nb = (int)block;
    int32_t *lam = fsm, *g1 = lam + block, *newF = g1 + ng1;
    uint16_t *sp = (uint16_t *)(newF + NEWF_CAP), *tp = sp + block + 2, *se = tp + block + 2, *te = se + cap;
    // a thread's consecutive points: entries inside the block, counted, then gathered
    const int per = nb / LT, t0 = tid * per;
    int s_sum = 0, t_sum = 0;
    for (int t = t0; t < t0 + per; ++t) {
        int cnt = 0, ns = 0;
        if (t < m) {
            const int64_t i = lo + t;
            for (int64_t a = strp[i]; a < strp[i + 1]; ++a) cnt += (stci[a] >= lo && stci[a] < hi);
            for (int64_t a = srp[i]; a < srp[i + 1]; ++a) ns += (sci[a] >= lo && sci[a] < hi);
        }
        lam[t] = cnt == 0 && ns == 0 ? LAM_F : cnt;
        s_sum += ns;
        t_sum += cnt;
    }
    // first entries of the thread's points: an inclusive scan in the warp, then over the warps
    int s_in = s_sum, t_in = t_sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int so = __shfl_up_sync(FULL, s_in, d), to = __shfl_up_sync(FULL, t_in, d);
        if (lane >= d) {
            s_in += so;
            t_in += to;
        }
    }
    if (lane == 31) {
        sum[0][tid >> 5] = s_in;
        sum[1][tid >> 5] = t_in;
    }
    __syncthreads();
    int s_at = s_in - s_sum, t_at = t_in - t_sum, total = 0;
    for (int u = 0; u < LT / 32; ++u) {
        if (u < (tid >> 5)) {
            s_at += sum[0][u];
            t_at += sum[1][u];
        }
        total += sum[0][u];                            // = the entries of S^T inside the block
    }
    const bool fits = total <= cap;
    if (fits) {
        for (int t = t0; t < t0 + per; ++t) {
            sp[t] = (uint16_t)s_at;
            tp[t] = (uint16_t)t_at;
            if (t < m) {
                const int64_t i = lo + t;
                for (int64_t a = srp[i]; a < srp[i + 1]; ++a)
                    if (sci[a] >= lo && sci[a] < hi) se[s_at++] = (uint16_t)(sci[a] - lo);
                for (int64_t a = strp[i]; a < strp[i + 1]; ++a)
                    if (stci[a] >= lo && stci[a] < hi) te[t_at++] = (uint16_t)(stci[a] - lo);
            }
        }
        if (tid == LT - 1) {
            sp[nb] = (uint16_t)s_at;
            tp[nb] = (uint16_t)t_at;
        }
    }
    for (int q = tid >> 5; q < ng1; q += LT / 32) {
        const int mx = __reduce_max_sync(FULL, lam[q * 32 + lane]);
        if (lane == 0) g1[q] = mx;
    }
    __syncthreads();
    if (tid < 32) {
        const LocalGraph g{lo, m, srp, strp, sci, stci, sp, tp, se, te};
        if (fits) local_picks<true>(g, ng1, lam, g1, newF, err);
        else local_picks<false>(g, ng1, lam, g1, newF, err);
    }
    __syncthreads();
    for (int t = tid; t < m; t += LT) cf[lo + t] = lam[t] == LAM_C ? CF_C : CF_F;
}

__device__ __forceinline__ double hash_frac(uint64_t x) {
    uint64_t z = x + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z = z ^ (z >> 31);
    return (double)(z >> 11) * (1.0 / 9007199254740992.0);
}

__device__ __forceinline__ double weight(const int64_t *strp, int64_t i) {
    return __dadd_rn((double)(strp[i + 1] - strp[i]), hash_frac((uint64_t)i));
}

__device__ __forceinline__ bool has_c(const int64_t *srp, const int32_t *sci, const int8_t *cf, int64_t i) {
    for (int64_t a = srp[i]; a < srp[i + 1]; ++a)
        if (cf[sci[a]] == CF_C) return true;
    return false;
}

__global__ void interface_init_kernel(int64_t n, int64_t block, const int64_t *srp, const int32_t *sci,
                                      const int64_t *strp, const int32_t *stci, const int8_t *cf, int8_t *inU,
                                      unsigned long long *count) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        int8_t u = 0;
        if (cf[i] == CF_F && srp[i + 1] > srp[i] && !has_c(srp, sci, cf, i)) {
            const int64_t bi = i / block;
            bool cross = false;
            for (int64_t a = srp[i]; a < srp[i + 1] && !cross; ++a) cross = sci[a] / block != bi;
            for (int64_t a = strp[i]; a < strp[i + 1] && !cross; ++a) cross = stci[a] / block != bi;
            u = cross ? 1 : 0;
        }
        inU[i] = u;
        if (u) atomicAdd(count, 1ull);
    }
}

__global__ void interface_select_kernel(int64_t n, const int64_t *srp, const int32_t *sci, const int64_t *strp,
                                        const int32_t *stci, const int8_t *inU, int8_t *sel) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        int8_t s = 0;
        if (inU[i]) {
            const double wi = weight(strp, i);
            bool best = true;
            for (int64_t a = srp[i]; a < srp[i + 1] && best; ++a) {
                const int32_t j = sci[a];
                if (!inU[j]) continue;
                const double wj = weight(strp, j);
                if (wj > wi || (wj == wi && j < i)) best = false;
            }
            for (int64_t a = strp[i]; a < strp[i + 1] && best; ++a) {
                const int32_t j = stci[a];
                if (!inU[j]) continue;
                const double wj = weight(strp, j);
                if (wj > wi || (wj == wi && j < i)) best = false;
            }
            s = best ? 1 : 0;
        }
        sel[i] = s;
    }
}

__global__ void interface_apply_kernel(int64_t n, const int8_t *sel, int8_t *cf, int8_t *inU) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        if (sel[i]) {
            cf[i] = CF_C;
            inU[i] = 0;
        }
}

__global__ void interface_leave_kernel(int64_t n, const int64_t *srp, const int32_t *sci, const int8_t *cf,
                                       int8_t *inU, unsigned long long *count) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        if (!inU[i]) continue;
        if (has_c(srp, sci, cf, i)) inU[i] = 0;
        else atomicAdd(count, 1ull);
    }
}

}  // namespace

int air_falgout_split(int64_t n, int64_t block, const int64_t *srp, const int32_t *sci, const int64_t *strp,
                      const int32_t *stci, int8_t *cf, int *d_err, cudaStream_t s) {
    if (block < 32 || block % 1024 != 0) return AIR_ERR_INVALID_ARG;
    const int64_t nblk = (n + block - 1) / block;
    // entries of a block's graph in shared memory: six per point (HDG levels hold two to five inside a block), up to
    // what the shared memory and 16-bit row starts allow; other blocks read the graph from global memory
    const size_t fixed = (size_t)(block + block / 32 + NEWF_CAP) * sizeof(int32_t) +
                         2 * (size_t)(block + 2) * sizeof(uint16_t);
    if (block > 8192) return AIR_ERR_UNSUPPORTED;
    int64_t cap = (int64_t)((AIR_SMEM_OPTIN - 2048 - fixed) / (2 * sizeof(uint16_t)));   // 2048: the static arrays
    if (cap > 6 * block) cap = 6 * block;
    const size_t smem = fixed + 2 * (size_t)cap * sizeof(uint16_t);
    AIR_CUDA(air_smem_optin(local_pass_kernel));
    local_pass_kernel<<<air_counted((unsigned)nblk), LT, smem, s>>>(n, block, (int)cap, srp, sci, strp, stci, cf, d_err);
    AIR_LAUNCH();
    int8_t *inU = nullptr, *sel = nullptr;
    unsigned long long *count = nullptr;
    AIR_CUDA(air_dmalloc((void **)&inU, (size_t)n));
    AIR_CUDA(air_dmalloc((void **)&sel, (size_t)n));
    AIR_CUDA(air_dmalloc((void **)&count, sizeof(unsigned long long)));
    int st = AIR_OK;
    unsigned long long left = 0;
    if (cudaMemsetAsync(count, 0, sizeof(unsigned long long), s) != cudaSuccess) st = AIR_ERR_CUDA;
    if (st == AIR_OK) {
        interface_init_kernel<<<air_counted(grid_for(n, 256)), 256, 0, s>>>(n, block, srp, sci, strp, stci, cf, inU,
                                                                            count);
        if (cudaMemcpyAsync(&left, count, sizeof(left), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess)
            st = AIR_ERR_CUDA;
    }
    // every round makes the heaviest remaining point of each component of U a C point
    for (int64_t round = 0; st == AIR_OK && left > 0; ++round) {
        if (round > n) { st = AIR_ERR_DEVICE_TIMEOUT; break; }
        interface_select_kernel<<<air_counted(grid_for(n, 256)), 256, 0, s>>>(n, srp, sci, strp, stci, inU, sel);
        interface_apply_kernel<<<air_counted(grid_for(n, 256)), 256, 0, s>>>(n, sel, cf, inU);
        if (cudaMemsetAsync(count, 0, sizeof(unsigned long long), s) != cudaSuccess) { st = AIR_ERR_CUDA; break; }
        interface_leave_kernel<<<air_counted(grid_for(n, 256)), 256, 0, s>>>(n, srp, sci, cf, inU, count);
        if (cudaMemcpyAsync(&left, count, sizeof(left), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess)
            st = AIR_ERR_CUDA;
    }
    air_dfree(inU);
    air_dfree(sel);
    air_dfree(count);
    return st;
}
