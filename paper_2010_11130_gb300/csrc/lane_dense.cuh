// Small dense blocks, one per lane: a warp holds 32 b x b matrices in shared
// memory, entry (r, c) of lane l's matrix at m[(r b + c) LANE_LD + l], so every
// step of an elimination is one full FP64 instruction for 32 blocks.  (One
// warp per block leaves most lanes of each instruction idle and repeats the
// divisions; GB300 issues one FP64 warp instruction per SM in 16 cycles.)  Or one
// per group of lanes, row-major, with shorter chains (group_invert).
#pragma once

#include <stdint.h>

#include <math.h>

constexpr int LANE_LD = 33;     // lanes plus one: loads that walk the entries touch distinct banks

// |x| as an integer whose order is that of the magnitudes (0: NaN, which never is a pivot): comparing integers keeps
// the pivot search off the FP64 lanes.
__device__ __forceinline__ unsigned long long magnitude_key(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
    return b > 0x7ff0000000000000ull ? 0ull : b + 1ull;
}

// Copies the blocks first .. first + count - 1 (count <= 32) of src (b x b row-major each, transposed when tr) into
// the warp's layout; the lanes past count get the identity.
__device__ __forceinline__ void lane_load_blocks(const double *src, int64_t first, int count, int b, bool tr, double *m) {
    const int lane = threadIdx.x & 31, bb = b * b;
    for (int k = 0; k < 32; ++k)
        for (int t = lane; t < bb; t += 32) {
            const int r = t / b, c = t % b;
            m[(tr ? c * b + r : t) * LANE_LD + k] = k < count ? src[(first + k) * bb + t] : (r == c ? 1.0 : 0.0);
        }
    __syncwarp();
}

// Row of the largest magnitude in column c of lane's matrix at or below row c (ties -> smallest); -1: no pivot.
__device__ __forceinline__ int lane_pivot(const double *m, int b, int c) {
    unsigned long long best = 1ull;
    int r = -1;
    for (int rr = c; rr < b; ++rr) {
        const unsigned long long k = magnitude_key(m[(rr * b + c) * LANE_LD]);
        if (k > best) { best = k; r = rr; }
    }
    return r;
}

// Inverts the lane's matrix in place (m points at the lane's first entry) by Gauss-Jordan with partial pivoting: the
// operations, in order, of the elimination of [M | I] (row / pivot, then fma(-f, row, other row)).  b <= 11.  Returns
// false, and leaves garbage, if a pivot is zero.
__device__ __forceinline__ bool lane_invert(double *m, int b) {
    unsigned long long perm = 0ull;                  // 4 bits per column
    for (int c = 0; c < b; ++c) {
        const int r = lane_pivot(m, b, c);
        if (r < 0) return false;
        perm |= (unsigned long long)r << (4 * c);
        if (r != c)
            for (int t = 0; t < b; ++t) {
                const double x = m[(c * b + t) * LANE_LD];
                m[(c * b + t) * LANE_LD] = m[(r * b + t) * LANE_LD];
                m[(r * b + t) * LANE_LD] = x;
            }
        const double piv = m[(c * b + c) * LANE_LD];
        m[(c * b + c) * LANE_LD] = 1.0;
        for (int t = 0; t < b; ++t) m[(c * b + t) * LANE_LD] = __ddiv_rn(m[(c * b + t) * LANE_LD], piv);
        for (int rr = 0; rr < b; ++rr) {
            if (rr == c) continue;
            const double f = m[(rr * b + c) * LANE_LD];
            m[(rr * b + c) * LANE_LD] = 0.0;
            for (int t = 0; t < b; ++t)
                m[(rr * b + t) * LANE_LD] = __fma_rn(-f, m[(c * b + t) * LANE_LD], m[(rr * b + t) * LANE_LD]);
        }
    }
    for (int c = b - 1; c >= 0; --c) {               // the row swaps, undone on the columns
        const int r = (int)(perm >> (4 * c)) & 15;
        if (r == c) continue;
        for (int t = 0; t < b; ++t) {
            const double x = m[(t * b + c) * LANE_LD];
            m[(t * b + c) * LANE_LD] = m[(t * b + r) * LANE_LD];
            m[(t * b + r) * LANE_LD] = x;
        }
    }
    return true;
}

// The same inverse by a group of b lanes, lane j (of the group) keeping column j; m is the group's matrix, row-major, and
// f b doubles of its own, both in shared memory.  Every lane of the warp calls it, those without a matrix with j >= b.
// The operations on an entry, and their order, are lane_invert's; a step is a chain of b of them instead of b^2, and the
// divisions of a row are one instruction either way.
__device__ __forceinline__ bool group_invert(double *m, double *f, int b, int j) {
    unsigned long long perm = 0ull;
    bool ok = true;
    for (int c = 0; c < b; ++c) {
        unsigned long long best = 1ull;
        int r = -1;
        for (int rr = c; rr < b; ++rr) {
            const unsigned long long k = magnitude_key(m[rr * b + c]);
            if (k > best) { best = k; r = rr; }
        }
        ok = ok && r >= 0;
        __syncwarp();
        if (ok && j < b && r != c) {
            const double x = m[c * b + j];
            m[c * b + j] = m[r * b + j];
            m[r * b + j] = x;
        }
        if (ok) perm |= (unsigned long long)r << (4 * c);
        __syncwarp();
        if (j < b) f[j] = m[j * b + c];
        __syncwarp();
        if (ok && j < b) {
            const double v = __ddiv_rn(j == c ? 1.0 : m[c * b + j], f[c]);
            m[c * b + j] = v;
            for (int rr = 0; rr < b; ++rr)
                if (rr != c) m[rr * b + j] = __fma_rn(-f[rr], v, j == c ? 0.0 : m[rr * b + j]);
        }
        __syncwarp();
    }
    for (int c = b - 1; c >= 0; --c) {
        const int r = (int)(perm >> (4 * c)) & 15;
        if (ok && j < b && r != c) {
            const double x = m[j * b + c];
            m[j * b + c] = m[j * b + r];
            m[j * b + r] = x;
        }
    }
    __syncwarp();
    return ok;
}
