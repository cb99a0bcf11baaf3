// sell.cuh -- row sums of the multigrid operators in sliced ELL, shared by the kernels that run one
// phase per launch (solve.cu) and those that run many (persist.cu), so that both give the same bits.
//
// A slice is one warp's work: 32 / L rows, L = 2^lsh lanes per row (Sell::lsh). Lane l works on row
// l mod (32 / L) of the slice as its part l div (32 / L); part q holds the row's entries q, q + L,
// q + 2L, ..., entry q + tL at off + 32 t + l. The parts' sums are added by a fixed xor tree.
//
// In a level's matrix the entries of earlier colours ("lower") come first in every row, so that a
// sweep from x = 0 reads only those, and the residual after it only the others: see Range.
#pragma once

#include <cuda_bf16.h>

#include "internal.cuh"

namespace vemg {

// BF16 values widen to FP32 before they meet the vector; FP32 and FP64 values pass through
__device__ __forceinline__ float float_or_self(__nv_bfloat16 a) { return __bfloat162float(a); }
__device__ __forceinline__ float float_or_self(float a) { return a; }
__device__ __forceinline__ double float_or_self(double a) { return a; }

struct SellView {
    const int4 *meta;      // per slice: first row, rows, element offset
    const unsigned *rl;    // per row: lower entries and entries (Sell::rl)
    const int *col;
    int lsh, rl_wide;
};

inline SellView view(const Sell &S) { return SellView{S.meta, S.rl, S.col, S.lsh, S.rl_wide}; }

// the part of each row that an operation takes
enum Range : int { ROW_ALL = 0, ROW_LOWER = 1, ROW_UPPER = 2 };

// a lane's share of a row: entries o + 32 t, t0 <= t < t1
struct LaneRow {
    int r, o, t0, t1;
    bool on, first;   // a row of the slice; the lane that stores the row's result
};

__device__ __forceinline__ LaneRow lane_row(const SellView &S, int s, int lane, int range) {
    const int4 m = __ldg(S.meta + s);
    const int rows = 32 >> S.lsh, k = lane & (rows - 1), q = lane >> (5 - S.lsh), up = (1 << S.lsh) - 1 - q;
    LaneRow a;
    a.on = k < m.y;
    a.first = a.on && q == 0;
    a.r = m.x + k;
    a.o = m.z + lane;
    a.t0 = a.t1 = 0;
    if (a.on) {
        unsigned lo, len;
        if (S.rl_wide) {
            lo = __ldg(S.rl + 2 * (int64_t)a.r);
            len = __ldg(S.rl + 2 * (int64_t)a.r + 1);
        } else {
            const unsigned w = __ldg(S.rl + a.r);
            lo = w & 0xffffu;
            len = w >> 16;
        }
        if (range == ROW_UPPER) a.t0 = ((int)lo + up) >> S.lsh;
        a.t1 = ((int)(range == ROW_LOWER ? lo : len) + up) >> S.lsh;
    }
    return a;
}

// The lane's first U entries (column indices and values), loaded before the kernel waits for its
// predecessor: the operators are setup data that no solve kernel writes, so these loads overlap the
// previous kernel and only the gathers of x remain after the wait.
template <class VT, int U>
struct RowHead {
    int c[U];
    VT a[U];
};

template <class VT, int U>
__device__ __forceinline__ void load_head(RowHead<VT, U> &h, const int *__restrict__ col, const VT *__restrict__ v,
                                          const LaneRow &a, int t) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
        h.c[u] = t + u < a.t1 ? __ldg(col + a.o + 32 * (t + u)) : 0;
        h.a[u] = t + u < a.t1 ? __ldg(v + a.o + 32 * (t + u)) : VT{};
    }
}

// one element of x: default caching, or through L2 where other CTAs of the same kernel write x
template <bool CG, class XT>
__device__ __forceinline__ XT load_x(const XT *x) {
    return CG ? __ldcg(x) : *x;
}

// the lane's share of the row's dot product with x: the head's entries, then the rest U at a time
// (columns and values first, then the gathers); products are added in entry order whatever U is
template <bool CG, class AT, class VT, class XT, int U>
__device__ __forceinline__ AT lane_sum(RowHead<VT, U> &h, const int *__restrict__ col, const VT *__restrict__ v,
                                       const LaneRow &a, const XT *x) {
    AT acc = 0;
    for (int t = a.t0;;) {
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (t + u < a.t1) acc = fmadd((AT)float_or_self(h.a[u]), (AT)load_x<CG>(x + h.c[u]), acc);
        t += U;
        if (t >= a.t1) return acc;
        load_head(h, col, v, a, t);
    }
}

// sum over the lanes of each row (all 32 lanes of the warp call it)
template <class AT>
__device__ __forceinline__ AT row_sum(AT acc, int lsh) {
    for (int o = 16; o >= (32 >> lsh); o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    return acc;
}

}  // namespace vemg
