// batch.cu -- many right-hand sides in one solve.
//
// K systems A x_c = b_c share one hierarchy. Vectors are interleaved (row-major n x K, K a power
// of two): x[i*K + c], in the natural (internal) ordering of each level. A group of KW lanes works on
// one row, each lane on V neighbouring columns per load (16 bytes where the batch is wide enough), so
// each matrix entry is read once for all columns and a gather of x[j*K ..] is one wide load per lane.
// Natural order keeps a row's neighbours close in memory, so the gathers stay in L2 even when the
// K-column vectors are far larger than L2 (the colour-major order of the one-column solve does
// not: each colour's pass would sweep the whole vector). Colour sweeps walk the level's list of
// rows of each colour. Each column keeps its own Krylov scalars
// (alpha, beta, norms, mean) and its own convergence test; a converged column is frozen (alpha = 0)
// until every column has converged. The iteration runs as CUDA graphs with a WHILE node, like the
// single right-hand-side solve (solve.cu); the V-cycles of the two branches run on two streams.
#include <math.h>

#include <algorithm>
#include <cstring>

#include <type_traits>
#include <vector>

#include "sell.cuh"

namespace vemg {

static constexpr int kBT = 512;        // threads of the streaming kernels
static constexpr int kMaxK = 128;      // widest batch
static constexpr int kSellWarps = 4;   // warps per block of the batched row kernels (untuned default)
static constexpr int kMaxWarps = 8;    // most warps per block the autotuner tries

static thread_local int64_t *b_count = nullptr;
struct BTune;
static thread_local const BTune *b_tune = nullptr;   // launch shapes of the batch being recorded

struct TuneScope {
    const BTune *saved;
    explicit TuneScope(const BTune *t) : saved(b_tune) { b_tune = t; }
    ~TuneScope() { b_tune = saved; }
};
#define BATCH_LAUNCHED()         \
    do {                         \
        VEMG_CHECK_LAUNCH();     \
        if (b_count) ++*b_count; \
    } while (0)

// per-column scalar slots (sc[slot * K + c])
enum {
    B_RZ = 0, B_PQ, B_ALPHA, B_BETA, B_MU, B_BN, B_RN, B_FLAG, B_ITERS, B_CONV, B_ZERO, B_TRUE, B_BMEAN, B_XMEAN,
    B_TOL, B_MAXIT, B_FRESH, B_BEST, B_LASTIMP, B_STALL, B_SUMR, B_SUMQ, B_COUNT
};

// a column whose best residual has not dropped by 1% in this many iterations has reached the
// round-off floor: it stops (status VEMG_ENOTCONV with its last residual)
static constexpr int kStallIters = 30;
// global scalars after the per-column block (g[slot])
enum { G_TOL = 0, G_MAXIT, G_CONT, G_ITERS, G_COUNT };

// One operator as the batched row kernels read it: entries of row r at rp[r] - r * diag, a row
// without its diagonal having one fewer (diag = 1). The chains' operators have their own copies:
// FP32 values packed with their columns (ent: 8 bytes an entry, one load), and in a level's matrix the
// diagonal left out and the entries of earlier colours first (lo[r] of them), so that a sweep from
// x = 0 reads only those and the residual after it only the others (as in the one-column solve).
struct BRows {
    const int *rp = nullptr, *ci = nullptr;
    const void *v = nullptr;
    const int2 *ent = nullptr;
    const int *lo = nullptr;
    const int4 *info = nullptr;   // a level's matrix: row, first entry, lower entries, entries; in sweep order
    int diag = 0;
    int qsh = 0;            // log2 of the parts a row is split into (parts_shift)
};

// one multigrid level as the batched cycle sees it
struct BLevel {
    int n = 0, ncolours = 0;
    const void *dinv = nullptr;
    std::vector<int> cptr;
    BRows A, P, PT;
};

struct BChain {
    int nlev = 0;
    BLevel lv[kMaxLevels];
    bool direct = false;
    int nc = 0;
    const double *G = nullptr;
    const float *Gf = nullptr;   // FP32 copy (FP32 cycles)
};

struct BatchGraphs {
    cudaGraph_t g = nullptr;
    cudaGraphExec_t exec = nullptr;
    cudaGraphConditionalHandle handle = 0;
    int64_t k_pre = 0, k_body = 0, k_post = 0;
};

// Launch shapes of the batched row kernels, by class: 0 = colour sweeps, 1 = the other V-cycle
// operations (residuals, restrictions, prolongations, E~ in FP32), 2 = the outer FP64 operations (A p,
// the true residual, E~ and E~^T). kw: lanes per row (each lane takes 16 bytes of neighbouring
// columns at a time), warps: warps per block. Chosen per batch width by timing the candidates (autotune below); the
// per-column arithmetic is the same for every shape.
struct BTune {
    int kw[3] = {0, 0, 0}, warps[3] = {0, 0, 0};   // 0: the untuned default
    float us[3] = {0.f, 0.f, 0.f};                  // the chosen shapes' measured launch times
    int tried = 0;                                   // candidate launches timed
};

struct BatchWork {
    BTune tune;
    int K = 0;
    double *X = nullptr, *R = nullptr, *Z = nullptr, *P = nullptr, *Q = nullptr, *B = nullptr;
    void *lx[2][kMaxLevels] = {}, *lb[2][kMaxLevels] = {}, *lr[2][kMaxLevels] = {};
    double *sc = nullptr;      // B_COUNT * K per-column scalars, then G_COUNT globals
    double *part = nullptr;    // reduction partials
    unsigned *ctr = nullptr;
    BatchGraphs *graphs = nullptr;
    Arena arena;
    BChain *bsurf = nullptr, *bbar = nullptr;
    BRows Aout, E, ET;   // the outer operators, FP64 (E: FP32 with FP32 V-cycles)
    const int *caller_of = nullptr;   // caller id of each unknown (internal order)
    // FP32 V-cycles: an FP32 copy of the A_bar part of the outer residual (the finest level's
    // right-hand side, converted once per application instead of on every read); E~'s values are
    // FP32 too (the prolongation z = E~ y_s is formed in FP32)
    float *Rb32 = nullptr;
    ~BatchWork() {
        delete bsurf;
        delete bbar;
    }
};

static double *gsc(BatchWork *w) { return w->sc + B_COUNT * w->K; }

// ------------------------------------------------------------------------------------------
// batched row operations (natural order)

// BOP_SPMV_PLUS: y = b_part + A x, where rows r >= cur start from b[(r - cur) K + c] (and the
// others from 0): z = [0; x_bar] + E~ y_s formed in the accumulator type, converted once.
// BOP_UPPER: the residual after a sweep from zero in ascending colours, y = -(entries of later colours) x
enum { BOP_SPMV = 0, BOP_SPMV_ADD = 1, BOP_SOR = 2, BOP_RES = 3, BOP_SPMV_PLUS = 4, BOP_UPPER = 5 };


// V neighbouring columns, in loads and stores of up to 16 bytes (p is aligned to V elements: V
// divides K and the vectors start on 256-byte boundaries)
template <int V, class T>
__device__ __forceinline__ void load_cols(const T *p, T (&o)[V]) {
    constexpr int B = V * (int)sizeof(T);
    if constexpr (B >= 16) {
#pragma unroll
        for (int k = 0; k < B / 16; ++k) {
            const float4 f = *(const float4 *)((const char *)p + 16 * k);
            memcpy((char *)o + 16 * k, &f, 16);
        }
    } else if constexpr (B == 8) {
        const float2 f = *(const float2 *)p;
        memcpy(o, &f, 8);
    } else {
        o[0] = *p;
    }
}
template <int V, class T>
__device__ __forceinline__ void store_cols(T *p, const T (&o)[V]) {
    constexpr int B = V * (int)sizeof(T);
    if constexpr (B >= 16) {
#pragma unroll
        for (int k = 0; k < B / 16; ++k) {
            float4 f;
            memcpy(&f, (const char *)o + 16 * k, 16);
            *(float4 *)((char *)p + 16 * k) = f;
        }
    } else if constexpr (B == 8) {
        float2 f;
        memcpy(&f, o, 8);
        *(float2 *)p = f;
    } else {
        *p = o[0];
    }
}

// up to kBU entries of a row
static constexpr int kBU = 4;
template <bool PACK, class VT>
struct Entries {
    int c[kBU];
    VT v[kBU];
    __device__ __forceinline__ void load(const BRows &A, int at, int step, int n) {
#pragma unroll
        for (int u = 0; u < kBU; ++u) {
            c[u] = 0;
            v[u] = (VT)0;
            if (u < n) {
                if constexpr (PACK) {
                    const int2 e = __ldg(A.ent + at + u * step);
                    c[u] = e.x;
                    v[u] = __int_as_float(e.y);
                } else {
                    c[u] = __ldg(A.ci + at + u * step);
                    v[u] = __ldg((const VT *)A.v + at + u * step);
                }
            }
        }
    }
};

// Rows idx in [0, nrows) (info: in sweep order, else in row order). A warp holds 32 / (KW Q) rows,
// KW = 1 << kwsh lanes by Q = 1 << A.qsh parts a row: lane l takes the columns (l mod KW) V + j KW V .. + V
// in pass j, part q the entries q, q + Q, ... of the row, and the parts are added by a fixed xor tree.
// The sum of a column thus depends on Q and not on the launch shape. K is a multiple of KW V.
//
// Latency of the gathers bounds it: 16-byte loads, four entries' gathers before their multiply-adds
// and the next four entries under way meanwhile, in at most 64 registers (four blocks of 8 warps per
// SM). The finest sweep's largest colour on the 384 x 384 x 24 mesh with 64 columns: 331 us (422 with one
// column per load). Eight columns a lane with eight entries held took 102 registers and 446 us; three,
// five or six blocks per SM, or two entries at a time, were slower for one batch width or another. The
// outer product is bound by the FP64 pipe instead (54.5M entries x 64 columns: 5.5 of its 6.3 ms).
template <int OP, bool PACK, class VT, class XT, class BT, class YT, class AT, int V>
__global__ void __launch_bounds__(32 * kMaxWarps, 4) k_brow(int nrows, const int4 *__restrict__ info, BRows A, int range,
                                                            const XT *__restrict__ dg, const BT *__restrict__ b,
                                                            const XT *x, YT *y, int K, int kwsh, int cur) {
    const int w = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    const int gsh = kwsh + A.qsh, rw = 32 >> gsh, kw = 1 << kwsh, Q = 1 << A.qsh;
    if ((int64_t)w * rw >= nrows) {   // warp-uniform
        pdl_begin();
        return;
    }
    const int idx = w * rw + (lane >> gsh), gl = lane & (kw - 1), part = (lane >> kwsh) & (Q - 1);
    const bool valid = idx < nrows, out = valid && part == 0;
    int r = 0, at = 0, n = 0;   // row, first entry and entries of this part
    if (valid) {
        int lo = 0, len;
        if (info) {
            const int4 m = __ldg(info + idx);
            r = m.x;
            at = m.y;
            lo = m.z;
            len = m.w;
        } else {
            r = idx;
            const int o = __ldg(A.rp + r);
            len = __ldg(A.rp + r + 1) - o - A.diag;
            if (range != ROW_ALL) lo = __ldg(A.lo + r);
            at = o - r * A.diag;
        }
        const int e0 = range == ROW_UPPER ? lo : 0, e1 = range == ROW_LOWER ? lo : len;
        at += e0 + part;
        n = (e1 - e0 - part + Q - 1) >> A.qsh;
    }
    Entries<PACK, VT> h;
    h.load(A, at, Q, n);
    const XT d = OP == BOP_SOR && out ? __ldg(dg + r) : (XT)0;
    pdl_begin();
    for (int c0 = gl * V; c0 < K; c0 += kw * V) {
        AT acc[V];
#pragma unroll
        for (int i = 0; i < V; ++i) acc[i] = (AT)0;
        BT bv[V];
        if ((OP == BOP_SOR || OP == BOP_RES) && out) load_cols<V>(b + (int64_t)r * K + c0, bv);
        if (OP == BOP_SPMV_PLUS && out && r >= cur) {
            load_cols<V>(b + (int64_t)(r - cur) * K + c0, bv);
#pragma unroll
            for (int i = 0; i < V; ++i) acc[i] = (AT)bv[i];
        }
        const XT *xc = x + c0;
        for (int t = 0; t < n; t += kBU) {
            XT g[kBU][V];
#pragma unroll
            for (int u = 0; u < kBU; ++u)
                if (t + u < n) load_cols<V>(xc + (int64_t)h.c[u] * K, g[u]);
            Entries<PACK, VT> cu = h;
            // the next entries of the row, or its first ones again for the next pass
            if (t + kBU < n) h.load(A, at + (t + kBU) * Q, Q, n - t - kBU);
            else if (n > kBU) h.load(A, at, Q, n);
#pragma unroll
            for (int u = 0; u < kBU; ++u)
                if (t + u < n)
#pragma unroll
                    for (int i = 0; i < V; ++i) acc[i] = fmadd((AT)cu.v[u], (AT)g[u][i], acc[i]);
        }
        for (int o = 1 << (gsh - 1); A.qsh > 0 && o >= kw; o >>= 1)
#pragma unroll
            for (int i = 0; i < V; ++i) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], o);
        if (!out) continue;
        const int64_t e = (int64_t)r * K + c0;
        YT res[V];
        if (OP == BOP_SPMV_ADD) load_cols<V>((const YT *)y + e, res);
#pragma unroll
        for (int i = 0; i < V; ++i) {
            const AT s = acc[i];
            if (OP == BOP_SPMV || OP == BOP_SPMV_PLUS) res[i] = cvt<YT>(s);
            else if (OP == BOP_SPMV_ADD) res[i] = (YT)((AT)res[i] + s);
            else if (OP == BOP_SOR) res[i] = (YT)((cvt<AT>(bv[i]) - s) * (AT)d);
            else if (OP == BOP_RES) res[i] = (YT)((AT)bv[i] - s);
            else res[i] = (YT)((AT)0 - s);
        }
        store_cols<V>(y + e, res);
    }
}

// V: the columns of a 16-byte load of x, where a lane has that many. kw, nw > 0 force a shape
// (autotuning); cls: the launch-shape class (BTune). info: the rows of a colour, else all rows.
template <int OP, bool PACK, class VT, class XT, class BT, class YT, class AT>
static void brow(const BRows &A, int nrows, const int4 *info, int range, const XT *dg, const BT *b, const XT *x, YT *y,
                 int K, int cur, cudaStream_t s, int cls = 1, int kw = 0, int nw = 0) {
    if (nrows <= 0) return;
    if (kw <= 0 && b_tune && b_tune->kw[cls] > 0) {
        kw = b_tune->kw[cls];
        nw = b_tune->warps[cls];
    }
    constexpr int VM = 16 / (int)sizeof(XT);
    const int wpb = nw > 0 ? nw : kSellWarps;
    if (kw <= 0) kw = K < 4 ? 1 : 32;
    const int KW = std::min(K, kw), V = std::min(K / KW, VM);
    int kwsh = 0;
    while ((1 << kwsh) < KW) ++kwsh;
    const int64_t per = 32 >> (kwsh + A.qsh), warps = (nrows + per - 1) / per;
    auto go = [&](auto v) {
        pdl_launch(k_brow<OP, PACK, VT, XT, BT, YT, AT, decltype(v)::value>, (int)((warps + wpb - 1) / wpb), 32 * wpb,
                   s, nrows, info, A, range, dg, b, x, y, K, kwsh, cur);
    };
    if (V == 1) go(std::integral_constant<int, 1>{});
    else if (V < VM) go(std::integral_constant<int, 2>{});
    else go(std::integral_constant<int, VM>{});
    BATCH_LAUNCHED();
}

// x = G b on the coarsest level: one block per row, its threads K columns by 256 / K parts of the row
static constexpr int kDenseThreads = 256;
template <class XT, class BT>
__global__ void __launch_bounds__(kDenseThreads) k_bdense(int n, const XT *__restrict__ G, const BT *__restrict__ b,
                                                          XT *__restrict__ x, int K) {
    pdl_begin();
    __shared__ XT sh[kDenseThreads];
    const int r = blockIdx.x, t = threadIdx.x, c = t & (K - 1), part = t / K, parts = kDenseThreads / K;
    XT s = 0;
#pragma unroll 8
    for (int j = part; j < n; j += parts) s = fmadd(__ldg(G + (int64_t)r * n + j), cvt<XT>(b[(int64_t)j * K + c]), s);
    sh[t] = s;
    for (int o = kDenseThreads / 2; o >= K; o >>= 1) {
        __syncthreads();
        if (t < o) sh[t] += sh[t + o];
    }
    __syncthreads();
    if (t < K) x[(int64_t)r * K + t] = sh[t];
}

// the chains' operators in FP32 are packed
template <class XT>
constexpr bool packed() { return sizeof(XT) == sizeof(float); }

template <class XT, class BT>
static void bsweep(const BLevel &L, const BT *b, XT *x, bool forward, bool from_zero, int K, cudaStream_t s) {
    for (int cc = 0; cc < L.ncolours; ++cc) {
        int c = forward ? cc : L.ncolours - 1 - cc;
        int nrows = L.cptr[c + 1] - L.cptr[c];
        brow<BOP_SOR, packed<XT>(), XT, XT, BT, XT, XT>(L.A, nrows, L.A.info + L.cptr[c],
                                                        from_zero ? ROW_LOWER : ROW_ALL, (const XT *)L.dinv, b, x, x,
                                                        K, -1, s, 0);
    }
}

// an event recorded where the cycle of a chain enters a level (k_blate's start)
struct BMark {
    const BChain *C = nullptr;
    int level = 0;
    cudaEvent_t ev = nullptr;
};
static thread_local BMark b_mark;

template <class XT, class BT>
static void bvcycle(const BChain &C, BatchWork *W, int ch, int l, const BT *b, XT *x, cudaStream_t s) {
    const BLevel &L = C.lv[l];
    const int K = W->K;
    if (b_mark.C == &C && l == b_mark.level) VEMG_CHECK_CUDA(cudaEventRecord(b_mark.ev, s));
    if (l == C.nlev - 1) {
        if (C.direct) {
            const XT *G = sizeof(XT) == sizeof(float) ? (const XT *)C.Gf : (const XT *)C.G;
            pdl_launch(k_bdense<XT, BT>, C.nc, kDenseThreads, s, C.nc, G, b, x, K);
            BATCH_LAUNCHED();
            return;
        }
        bsweep<XT, BT>(L, b, x, true, true, K, s);
        bsweep<XT, BT>(L, b, x, false, false, K, s);
        return;
    }
    constexpr bool P = packed<XT>();
    XT *r = (XT *)W->lr[ch][l];
    XT *nb = (XT *)W->lb[ch][l + 1], *nx = (XT *)W->lx[ch][l + 1];
    const BLevel &N = C.lv[l + 1];
    const XT *none = nullptr;
    bsweep<XT, BT>(L, b, x, true, true, K, s);
    // a warp's rows end together in sweep order (rows of one colour have about as many entries of later
    // ones): used while the vector stays in L2 over the passes of the colours; else in row order
    const bool sweep_order = (double)L.n * K * sizeof(XT) <= 64.0 * 1048576.0;
    brow<BOP_UPPER, P, XT, XT, XT, XT, XT>(L.A, L.n, sweep_order ? L.A.info : nullptr, ROW_UPPER, none, none, x, r, K,
                                           -1, s);
    brow<BOP_SPMV, P, XT, XT, XT, XT, XT>(L.PT, N.n, nullptr, ROW_ALL, none, none, r, nb, K, -1, s);
    bvcycle<XT, XT>(C, W, ch, l + 1, (const XT *)nb, nx, s);
    brow<BOP_SPMV_ADD, P, XT, XT, XT, XT, XT>(L.P, L.n, nullptr, ROW_ALL, none, none, nx, x, K, -1, s);
    bsweep<XT, BT>(L, b, x, false, false, K, s);
}

// ------------------------------------------------------------------------------------------
// per-column deterministic reductions in two stages. Stage 1 (streaming kernels): the blocks
// stride over the n x K block by kBT * kBE elements; thread t always holds column
// t % K (K divides kBT), loads a trip's elements first, and the block writes one partial per
// column and sum. Stage 2 (k_bstage2): one block per column adds the block partials in fixed
// order and applies the scalar step of that column; the last column block sets the globals.

static constexpr int kBE = 4;   // elements per thread and trip in stage 1

// blocks of stage 1: two per SM (fewer for a small batch), each in trips of kBT * kBE elements; partials
// stay few for stage 2 (one block per 4,096 elements wrote and read 150 MB of them at n K = 2.4e8)
static int stage1_blocks(int64_t N) {
    return (int)std::min<int64_t>(304, (N + (int64_t)kBT * kBE - 1) / ((int64_t)kBT * kBE));
}

template <int NS>
__device__ void bblock_partials(double (&acc)[NS], int K, double *part) {
    __shared__ double sh[kBT];
    const int t = threadIdx.x;
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        sh[t] = acc[s];
        __syncthreads();
        if (t < K) {
            double v = 0.0;
            for (int j = t; j < kBT; j += K) v += sh[j];
            part[((int64_t)blockIdx.x * NS + s) * K + t] = v;
        }
        __syncthreads();
    }
}

// stage-1 sum of a * b per column (b null: of a)
__global__ void __launch_bounds__(kBT) k_bsum(int64_t N, int K, const double *a, const double *b, double *part) {
    pdl_begin();
    double acc[1] = {0.0};
    for (int64_t base = (int64_t)blockIdx.x * kBT * kBE + threadIdx.x; base < N; base += (int64_t)gridDim.x * kBT * kBE) {
        double va[kBE], vb[kBE];
#pragma unroll
        for (int j = 0; j < kBE; ++j) {
            int64_t e = base + (int64_t)j * kBT;
            va[j] = e < N ? a[e] : 0.0;
            vb[j] = (e < N && b) ? b[e] : 1.0;
        }
#pragma unroll
        for (int j = 0; j < kBE; ++j) acc[0] = fma(va[j], vb[j], acc[0]);
    }
    bblock_partials<1>(acc, K, part);
}

// the preconditioner's sums over z, r (and q): s0 = sum z, s1 = sum r z [, s2 = sum z q] (k_blate has those
// of r and q); each vector is loaded once per element. FP64 and memory bound it: a multiply-add a sum
// (one: 1.0, see dadd).
template <int NS>
__global__ void __launch_bounds__(kBT, 2) k_bsums_zrq(int64_t N, int K, const double *__restrict__ z,
                                                      const double *__restrict__ r, const double *__restrict__ q,
                                                      double *part, double one) {
    pdl_begin();
    double acc[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) acc[s] = 0.0;
    for (int64_t base = (int64_t)blockIdx.x * kBT * kBE + threadIdx.x; base < N; base += (int64_t)gridDim.x * kBT * kBE) {
        double vz[kBE], vr[kBE], vq[kBE];
#pragma unroll
        for (int j = 0; j < kBE; ++j) {
            int64_t e = base + (int64_t)j * kBT;
            vz[j] = e < N ? z[e] : 0.0;
            vr[j] = e < N ? r[e] : 0.0;
            vq[j] = (NS == 3 && e < N) ? q[e] : 0.0;
        }
#pragma unroll
        for (int j = 0; j < kBE; ++j) {
            acc[0] = dadd(acc[0], vz[j], one);
            acc[1] = fma(vr[j], vz[j], acc[1]);
            if (NS == 3) acc[NS - 1] = fma(vz[j], vq[j], acc[NS - 1]);
        }
    }
    bblock_partials<NS>(acc, K, part);
}

enum { ST_MEAN_B = 0, ST_BN, ST_ALPHA, ST_RN, ST_BETA, ST_MEAN_X, ST_TRUE, ST_LATE };

// stage 2: one block per column, one warp per sum
__global__ void __launch_bounds__(256) k_bstage2(int op, int nblk, int ns, int K, const double *__restrict__ part,
                                                double *sc, double inv_n, int neumann, int flexible, int first,
                                                unsigned *ctr, int *active, cudaGraphConditionalHandle handle,
                                                int use_cond) {
    pdl_begin();
    __shared__ double tot[5];
    const int c = blockIdx.x, t = threadIdx.x, warp = t >> 5;
    if (warp < ns) {
        double v = 0.0;
        for (int k = t & 31; k < nblk; k += 32) v += part[((int64_t)k * ns + warp) * K + c];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if ((t & 31) == 0) tot[warp] = v;
    }
    __syncthreads();
    double *g = sc + B_COUNT * K;
    if (t == 0) {
        // converged, broken down, or out of iterations: frozen while other columns continue
        bool frozen = sc[B_CONV * K + c] != 0.0 || sc[B_FLAG * K + c] != 0.0 ||
                      sc[B_ITERS * K + c] >= sc[B_MAXIT * K + c] || sc[B_STALL * K + c] != 0.0;
        switch (op) {
            case ST_MEAN_B: sc[B_BMEAN * K + c] = tot[0] * inv_n; break;
            case ST_MEAN_X: sc[B_XMEAN * K + c] = tot[0] * inv_n; break;
            case ST_TRUE: sc[B_TRUE * K + c] = sqrt(tot[0]); break;
            case ST_LATE:
                sc[B_SUMR * K + c] = tot[0];
                if (ns > 1) sc[B_SUMQ * K + c] = tot[1];
                break;
            case ST_BN: {
                double bn = sqrt(tot[0]);
                sc[B_BN * K + c] = bn;
                if (bn == 0.0) {
                    sc[B_ZERO * K + c] = 1.0;
                    sc[B_CONV * K + c] = 1.0;
                } else if (sc[B_MAXIT * K + c] > 0.0) {
                    atomicOr(active, 1);
                }
                __threadfence();
                if (atomicAdd(ctr, 1u) == (unsigned)(K - 1)) {
                    g[G_CONT] = atomicAdd(active, 0) ? 1.0 : 0.0;
                    *active = 0;
                    *ctr = 0u;
                }
                break;
            }
            case ST_ALPHA: {
                double pq = tot[0];
                sc[B_PQ * K + c] = pq;
                if (frozen) sc[B_ALPHA * K + c] = 0.0;
                else if (!(pq > 0.0)) {
                    sc[B_FLAG * K + c] = 1.0;
                    sc[B_ALPHA * K + c] = 0.0;
                } else sc[B_ALPHA * K + c] = sc[B_RZ * K + c] / pq;
                break;
            }
            case ST_RN: {
                double rn = sqrt(tot[0]);
                if (!frozen) {
                    sc[B_RN * K + c] = rn;
                    sc[B_ITERS * K + c] += 1.0;
                    if (!(rn == rn)) sc[B_FLAG * K + c] = 1.0;
                    else if (rn <= sc[B_TOL * K + c] * sc[B_BN * K + c]) sc[B_CONV * K + c] = 1.0;
                    double best = sc[B_BEST * K + c];
                    if (best == 0.0 || rn < 0.99 * best) {
                        sc[B_BEST * K + c] = rn;
                        sc[B_LASTIMP * K + c] = sc[B_ITERS * K + c];
                    } else if (sc[B_ITERS * K + c] - sc[B_LASTIMP * K + c] >= kStallIters) {
                        sc[B_STALL * K + c] = 1.0;
                    }
                    if (sc[B_CONV * K + c] == 0.0 && sc[B_FLAG * K + c] == 0.0 && sc[B_STALL * K + c] == 0.0 &&
                        sc[B_ITERS * K + c] < sc[B_MAXIT * K + c])
                        atomicOr(active, 1);
                }
                __threadfence();
                if (atomicAdd(ctr, 1u) == (unsigned)(K - 1)) {
                    // last column: every other column's flag is visible
                    int act = atomicAdd(active, 0);
                    g[G_ITERS] += 1.0;
                    g[G_CONT] = act ? 1.0 : 0.0;
                    if (use_cond) cudaGraphSetConditional(handle, act ? 1u : 0u);
                    *active = 0;
                    *ctr = 0u;
                }
                break;
            }
            case ST_BETA: {
                double mu = neumann ? tot[0] * inv_n : 0.0;
                double rz = tot[1] - mu * sc[B_SUMR * K + c];
                double beta = 0.0;
                const bool fresh = sc[B_FRESH * K + c] != 0.0;
                sc[B_FRESH * K + c] = 0.0;
                if (!fresh && !frozen) {
                    if (flexible) beta = -(tot[2] - mu * sc[B_SUMQ * K + c]) / sc[B_PQ * K + c];
                    else beta = rz / sc[B_RZ * K + c];
                    if (!(rz == rz) || !(beta == beta)) sc[B_FLAG * K + c] = 1.0;
                }
                sc[B_MU * K + c] = mu;
                sc[B_BETA * K + c] = frozen ? 0.0 : beta;
                sc[B_RZ * K + c] = rz;
                break;
            }
        }
    }
}

// b -= mean (Neumann), r = b, x = p = 0 (streaming, no reduction)
// rb32 (FP32 V-cycles on two chains): the FP32 copy of r's A_bar part (elements from off32 on),
// the finest A_bar level's right-hand side; every kernel that writes r writes it too
__global__ void k_bprepare(int64_t N, int K, int neumann, double *__restrict__ b, double *__restrict__ r,
                           double *__restrict__ x, double *__restrict__ p, const double *__restrict__ sc,
                           float *__restrict__ rb32, int64_t off32) {
    int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= N) return;
    double bi = b[e] - (neumann ? sc[B_BMEAN * K + (int)(e & (K - 1))] : 0.0);
    b[e] = bi;
    r[e] = bi;
    if (rb32 && e >= off32) rb32[e - off32] = (float)bi;
    x[e] = 0.0;
    p[e] = 0.0;
}

// R -= alpha Q per column, the FP32 copy of R's A_bar part, and the stage-1 sums of R * R (elements of a
// thread and order as in k_bsum)
__global__ void __launch_bounds__(kBT, 2) k_bupdate_r(int64_t N, int K, const double *__restrict__ q,
                                                      double *__restrict__ r, const double *__restrict__ sc,
                                                      float *__restrict__ rb32, int64_t off32, double *part) {
    pdl_begin();
    double acc[1] = {0.0};
    const double a = sc[B_ALPHA * K + (int)(threadIdx.x & (K - 1))];   // kBT is a multiple of K: one column
    for (int64_t base = (int64_t)blockIdx.x * kBT * kBE + threadIdx.x; base < N; base += (int64_t)gridDim.x * kBT * kBE) {
        double vq[kBE], vr[kBE];
#pragma unroll
        for (int j = 0; j < kBE; ++j) {
            const int64_t e = base + (int64_t)j * kBT;
            if (e < N) { vq[j] = q[e]; vr[j] = r[e]; }
        }
#pragma unroll
        for (int j = 0; j < kBE; ++j) {
            const int64_t e = base + (int64_t)j * kBT;
            if (e >= N) continue;
            const double rn = fma(-a, vq[j], vr[j]);
            r[e] = rn;
            if (rb32 && e >= off32) rb32[e - off32] = cvt_f32(rn);
            acc[0] = fma(rn, rn, acc[0]);
        }
    }
    bblock_partials<1>(acc, K, part);
}

// What an iteration owes that nothing before the next z needs, on the side stream beside the coarse levels
// (as k_late of the one-column solve): X += alpha P and the stage-1 sums of R and, NS = 2, of Q. NS = 0:
// X alone. After any iteration the solution of a column is X + alpha P.
template <int NS>
__global__ void __launch_bounds__(kBT, 2) k_blate(int64_t N, int K, const double *__restrict__ p, double *__restrict__ x,
                                                  const double *__restrict__ r, const double *__restrict__ q,
                                                  const double *__restrict__ sc, double *part, double one) {
    pdl_begin();
    double acc[NS > 0 ? NS : 1] = {};
    const double a = sc[B_ALPHA * K + (int)(threadIdx.x & (K - 1))];
    for (int64_t base = (int64_t)blockIdx.x * kBT * kBE + threadIdx.x; base < N; base += (int64_t)gridDim.x * kBT * kBE) {
        double vp[kBE], vx[kBE], vr[kBE], vq[kBE];
#pragma unroll
        for (int j = 0; j < kBE; ++j) {
            const int64_t e = base + (int64_t)j * kBT;
            if (e >= N) continue;
            vp[j] = p[e];
            vx[j] = x[e];
            if (NS > 0) vr[j] = r[e];
            if (NS > 1) vq[j] = q[e];
        }
#pragma unroll
        for (int j = 0; j < kBE; ++j) {
            const int64_t e = base + (int64_t)j * kBT;
            if (e >= N) continue;
            x[e] = fma(a, vp[j], vx[j]);
            if (NS > 0) acc[0] = dadd(acc[0], vr[j], one);
            if (NS > 1) acc[NS - 1] = dadd(acc[NS - 1], vq[j], one);
        }
    }
    if constexpr (NS > 0) bblock_partials<NS>(acc, K, part);
}

// z += x (assign: z = x)
template <class XT>
__global__ void k_badd(int64_t N, const XT *__restrict__ x, double *__restrict__ z, int assign = 0) {
    pdl_begin();
    int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= N) return;
    z[e] = assign ? cvt<double>(x[e]) : z[e] + cvt<double>(x[e]);
}

// P = (Z - mu) + beta P per column
__global__ void k_bupdate_p(int64_t N, int K, const double *__restrict__ sc, const double *__restrict__ z,
                            double *__restrict__ p) {
    pdl_begin();
    int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= N) return;
    int c = (int)(e & (K - 1));
    p[e] = fma(sc[B_BETA * K + c], p[e], z[e] - sc[B_MU * K + c]);
}

__global__ void k_bsub_mean(int64_t N, int K, double *__restrict__ x, const double *__restrict__ sc, int slot) {
    int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e < N) x[e] -= sc[slot * K + (int)(e & (K - 1))];
}


__global__ void k_binit(double *sc, int K, double tol, int maxit) {
    for (int i = 0; i < B_COUNT * K + G_COUNT; ++i) sc[i] = 0.0;
    for (int c = 0; c < K; ++c) {
        sc[B_TOL * K + c] = tol;
        sc[B_MAXIT * K + c] = (double)maxit;
        sc[B_FRESH * K + c] = 1.0;
    }
    double *g = sc + B_COUNT * K;
    g[G_TOL] = tol;
    g[G_MAXIT] = (double)maxit;
}

// Between k caller-order columns (column c at [c * ld]) and the interleaved block, 32 rows by up to 32
// columns at a time through shared memory, so that both sides move whole sectors (the caller's order
// keeps runs of the internal one). The block's columns past k are zeros.
static constexpr int kTile = 32;

__global__ void __launch_bounds__(256) k_bgather(int nu, int K, int k, int64_t ldb, const int *__restrict__ caller_of,
                                                 const double *__restrict__ Bin, double *__restrict__ Bk) {
    __shared__ double tile[kTile][kTile + 1];
    const int i0 = blockIdx.x * kTile, c0 = blockIdx.y * kTile, W = min(K - c0, kTile);
    for (int e = threadIdx.x; e < kTile * W; e += 256) {
        const int i = e % kTile, c = e / kTile;
        tile[i][c] = i0 + i < nu && c0 + c < k ? Bin[(int64_t)(c0 + c) * ldb + caller_of[i0 + i]] : 0.0;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < kTile * W; e += 256) {
        const int i = e / W, c = e % W;
        if (i0 + i < nu) Bk[(int64_t)(i0 + i) * K + c0 + c] = tile[i][c];
    }
}

__global__ void __launch_bounds__(256) k_bscatter(int nu, int K, int k, int64_t ldx, const int *__restrict__ caller_of,
                                                  const double *__restrict__ Xk, double *__restrict__ Xout) {
    __shared__ double tile[kTile][kTile + 1];
    const int i0 = blockIdx.x * kTile, c0 = blockIdx.y * kTile, W = min(K - c0, kTile);
    for (int e = threadIdx.x; e < kTile * W; e += 256) {
        const int i = e / W, c = e % W;
        if (i0 + i < nu) tile[i][c] = Xk[(int64_t)(i0 + i) * K + c0 + c];
    }
    __syncthreads();
    for (int e = threadIdx.x; e < kTile * W; e += 256) {
        const int i = e % kTile, c = e / kTile;
        if (i0 + i < nu && c0 + c < k) Xout[(int64_t)(c0 + c) * ldx + caller_of[i0 + i]] = tile[i][c];
    }
}

// Dirichlet top: x = 0 on the top nodes
__global__ void k_btops(int ntop, int k, int64_t ldx, const int *__restrict__ tops, double *__restrict__ Xout) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t < (int64_t)ntop * k) Xout[(t / ntop) * ldx + tops[t % ntop]] = 0.0;
}

__global__ void k_bcond_init(const double *g, cudaGraphConditionalHandle handle) {
    cudaGraphSetConditional(handle, g[G_CONT] != 0.0 ? 1u : 0u);
}

// ------------------------------------------------------------------------------------------
// the batched iteration

static void bstage2(vemg_hierarchy *h, BatchWork *W, int op, int ns, int64_t N, int first, cudaStream_t s,
                    cudaGraphConditionalHandle hd = 0, int use_cond = 0) {
    pdl_launch(k_bstage2, W->K, 256, s, op, stage1_blocks(N), ns, W->K, (const double *)W->part, W->sc,
               1.0 / (double)h->nu, (int)(h->bc == VEMG_NEUMANN), (int)(h->precision != VEMG_PREC_FP64), first, W->ctr,
               (int *)(W->ctr + 1), hd, use_cond);
    BATCH_LAUNCHED();
}

// k_blate and its stage 2 on stream s (the cycle uses no partials)
static void blate(vemg_hierarchy *h, BatchWork *W, cudaStream_t s) {
    const int64_t N = (int64_t)h->nu * W->K;
    const bool flex = h->precision != VEMG_PREC_FP64;
    if (flex)
        pdl_launch(k_blate<2>, stage1_blocks(N), kBT, s, N, W->K, (const double *)W->P, W->X, (const double *)W->R,
                   (const double *)W->Q, (const double *)W->sc, W->part, 1.0);
    else
        pdl_launch(k_blate<1>, stage1_blocks(N), kBT, s, N, W->K, (const double *)W->P, W->X, (const double *)W->R,
                   (const double *)nullptr, (const double *)W->sc, W->part, 1.0);
    BATCH_LAUNCHED();
    bstage2(h, W, ST_LATE, flex ? 2 : 1, N, 0, s);
}

template <class XT>
static void bprecond(vemg_hierarchy *h, BatchWork *W, cudaStream_t s) {
    const int K = W->K;
    const bool two = !single_chain(h);
    const int mt = two ? h->mtop : 0;
    XT *xb = (XT *)W->lx[1][0];
    // k_blate starts where the A_bar cycle enters its first level of at most an eighth of the rows
    const BChain &B = *W->bbar;
    int lv = 0;
    while (lv + 1 < B.nlev && (int64_t)B.lv[lv].n * 8 > B.lv[0].n) ++lv;
    auto cycle = [&](auto *b) {
        b_mark = BMark{&B, lv, h->ev_mid};
        try {
            bvcycle<XT>(B, W, 1, 0, b, xb, s);
        } catch (...) {
            b_mark = BMark{};
            throw;
        }
        b_mark = BMark{};
        VEMG_CHECK_CUDA(cudaStreamWaitEvent(h->side, h->ev_mid, 0));
        blate(h, W, h->side);
        VEMG_CHECK_CUDA(cudaEventRecord(h->ev_join, h->side));
        VEMG_CHECK_CUDA(cudaStreamWaitEvent(s, h->ev_join, 0));
    };
    if (two) {
        XT *b0 = (XT *)W->lb[0][0], *x0 = (XT *)W->lx[0][0];
        VEMG_CHECK_CUDA(cudaEventRecord(h->ev_fork, s));
        VEMG_CHECK_CUDA(cudaStreamWaitEvent(h->side, h->ev_fork, 0));
        // surface branch: r_c = E~^T r in FP64, one V-cycle on E~^T A E~
        brow<BOP_SPMV, false, double, double, double, XT, double>(W->ET, h->mtop, nullptr, ROW_ALL,
                                                                  (const double *)nullptr, (const double *)nullptr,
                                                                  W->R, b0, K, -1, h->side, 2);
        bvcycle<XT, XT>(*W->bsurf, W, 0, 0, (const XT *)b0, x0, h->side);
        if constexpr (std::is_same<XT, float>::value) cycle((const float *)W->Rb32);   // kept current by every writer of r
        else cycle((const double *)W->R + (int64_t)mt * K);
        // z = E~ y_s + [0; x_bar]: with FP32 V-cycles formed in FP32 from x_bar on and converted
        // once into the FP64 z; with FP64 ones in FP64
        if constexpr (std::is_same<XT, float>::value) {
            brow<BOP_SPMV_PLUS, false, float, float, float, double, float>(W->E, h->n, nullptr, ROW_ALL,
                                                                           (const float *)nullptr, xb, x0, W->Z, K,
                                                                           mt, s, 1);
        } else {
            brow<BOP_SPMV, false, double, double, double, double, double>(W->E, h->n, nullptr, ROW_ALL,
                                                                          (const double *)nullptr,
                                                                          (const double *)nullptr, x0, W->Z, K, -1, s,
                                                                          2);
            const int64_t nbk = (int64_t)(h->n - mt) * K;
            pdl_launch(k_badd<XT>, grid_for(nbk, 256), 256, s, nbk, (const XT *)xb, W->Z + (int64_t)mt * K, 0);
            BATCH_LAUNCHED();
        }
    } else {
        cycle((const double *)W->R);
        int64_t N = (int64_t)h->nu * K;
        pdl_launch(k_badd<XT>, grid_for(N, 256), 256, s, N, (const XT *)xb, W->Z, 1);
        BATCH_LAUNCHED();
    }
}

// the first element of r's A_bar part (the FP32 copy covers it)
static int64_t rb32_offset(const vemg_hierarchy *h, const BatchWork *W) {
    return single_chain(h) ? 0 : (int64_t)h->mtop * W->K;
}

// one per-column sum (the wider sums of the preconditioner step are k_bsums_zrq's)
static void bsum(BatchWork *W, int64_t N, const double *a, const double *b, cudaStream_t s) {
    pdl_launch(k_bsum, stage1_blocks(N), kBT, s, N, W->K, a, b, W->part);
    BATCH_LAUNCHED();
}

static void bprecond_any(vemg_hierarchy *h, BatchWork *W, cudaStream_t s) {
    if (h->precision != VEMG_PREC_FP64) bprecond<float>(h, W, s);   // BF16 hierarchies: FP32 values here
    else bprecond<double>(h, W, s);
    // t0 = sum z, t1 = (r, z) [, t2 = (z, q)]
    int64_t N = (int64_t)h->nu * W->K;
    bool flex = h->precision != VEMG_PREC_FP64;
    const int ns = flex ? 3 : 2;
    if (flex)
        pdl_launch(k_bsums_zrq<3>, stage1_blocks(N), kBT, s, N, W->K, (const double *)W->Z, (const double *)W->R,
                   (const double *)W->Q, W->part, 1.0);
    else
        pdl_launch(k_bsums_zrq<2>, stage1_blocks(N), kBT, s, N, W->K, (const double *)W->Z, (const double *)W->R,
                   (const double *)nullptr, W->part, 1.0);
    BATCH_LAUNCHED();
    bstage2(h, W, ST_BETA, ns, N, 0, s);
}

// b -= mean (Neumann), r = b, x = p = 0, ||b|| per column; the iterations themselves start in the
// loop body, where every column enters as fresh (first direction p = z - mu)
static void bphase_pre(vemg_hierarchy *h, BatchWork *W, cudaStream_t s) {
    const int K = W->K, nu = h->nu;
    const int64_t N = (int64_t)nu * K;
    const bool neu = h->bc == VEMG_NEUMANN;
    if (neu) {
        bsum(W, N, W->B, nullptr, s);
        bstage2(h, W, ST_MEAN_B, 1, N, 0, s);
    }
    k_bprepare<<<grid_for(N, 256), 256, 0, s>>>(N, K, neu, W->B, W->R, W->X, W->P, W->sc, W->Rb32, rb32_offset(h, W));
    BATCH_LAUNCHED();
    bsum(W, N, W->B, W->B, s);
    bstage2(h, W, ST_BN, 1, N, 0, s);
}

static void bphase_step(vemg_hierarchy *h, BatchWork *W, cudaStream_t s, cudaGraphConditionalHandle hd, int use_cond) {
    const int K = W->K;
    const int64_t N = (int64_t)h->nu * K;
    brow<BOP_SPMV, false, double, double, double, double, double>(W->Aout, h->nu, nullptr, ROW_ALL,
                                                                  (const double *)nullptr, (const double *)nullptr,
                                                                  W->P, W->Q, K, -1, s, 2);
    {
        bsum(W, N, W->P, W->Q, s);
        bstage2(h, W, ST_ALPHA, 1, N, 0, s);
    }
    pdl_launch(k_bupdate_r, stage1_blocks(N), kBT, s, N, K, (const double *)W->Q, W->R, (const double *)W->sc, W->Rb32,
               rb32_offset(h, W), W->part);
    BATCH_LAUNCHED();
    bstage2(h, W, ST_RN, 1, N, 0, s, hd, use_cond);
}

static void bphase_direction(vemg_hierarchy *h, BatchWork *W, cudaStream_t s) {
    bprecond_any(h, W, s);
    int64_t N = (int64_t)h->nu * W->K;
    pdl_launch(k_bupdate_p, grid_for(N, 256), 256, s, N, W->K, (const double *)W->sc, (const double *)W->Z, W->P);
    BATCH_LAUNCHED();
}

static void bphase_post(vemg_hierarchy *h, BatchWork *W, cudaStream_t s) {
    const int K = W->K, nu = h->nu;
    const int64_t N = (int64_t)nu * K;
    pdl_launch(k_blate<0>, stage1_blocks(N), kBT, s, N, K, (const double *)W->P, W->X, (const double *)nullptr,
               (const double *)nullptr, (const double *)W->sc, W->part, 1.0);
    BATCH_LAUNCHED();
    if (h->bc == VEMG_NEUMANN) {
        bsum(W, N, W->X, nullptr, s);
        bstage2(h, W, ST_MEAN_X, 1, N, 0, s);
        k_bsub_mean<<<grid_for(N, 256), 256, 0, s>>>(N, K, W->X, W->sc, B_XMEAN);
        BATCH_LAUNCHED();
    }
    // true residual into Q
    brow<BOP_RES, false, double, double, double, double, double>(W->Aout, h->nu, nullptr, ROW_ALL,
                                                                 (const double *)nullptr, W->B, W->X, W->Q, K, -1, s,
                                                                 2);
    bsum(W, N, W->Q, W->Q, s);
    bstage2(h, W, ST_TRUE, 1, N, 0, s);
}

static void release_batch_graphs(BatchWork *W) {
    BatchGraphs *G = W->graphs;
    if (!G) return;
    if (G->exec) cudaGraphExecDestroy(G->exec);
    if (G->g) cudaGraphDestroy(G->g);
    delete G;
    W->graphs = nullptr;
}

static void build_batch_graphs(vemg_hierarchy *h, BatchWork *W) {
    BatchGraphs *G = new BatchGraphs();
    W->graphs = G;
    cudaStream_t cs;
    VEMG_CHECK_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
    int64_t *saved = b_count;
    int64_t count = 0;
    b_count = &count;
    try {
        // one graph per solve: the preparation and the kernel that sets the loop condition, a
        // WHILE node whose body is one iteration of every column, then the exit work
        VEMG_CHECK_CUDA(cudaGraphCreate(&G->g, 0));
        VEMG_CHECK_CUDA(cudaGraphConditionalHandleCreate(&G->handle, G->g, 0, cudaGraphCondAssignDefault));
        VEMG_CHECK_CUDA(cudaStreamBeginCaptureToGraph(cs, G->g, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
        bphase_pre(h, W, cs);
        k_bcond_init<<<1, 1, 0, cs>>>(gsc(W), G->handle);
        BATCH_LAUNCHED();
        G->k_pre = count;
        cudaStreamCaptureStatus st;
        const cudaGraphNode_t *deps = nullptr;
        size_t ndeps = 0;
        VEMG_CHECK_CUDA(cudaStreamGetCaptureInfo(cs, &st, nullptr, nullptr, &deps, nullptr, &ndeps));
        std::vector<cudaGraphNode_t> frontier(deps, deps + ndeps);
        cudaGraph_t captured = G->g;
        VEMG_CHECK_CUDA(cudaStreamEndCapture(cs, &captured));
        cudaGraphNodeParams cp = {};
        cp.type = cudaGraphNodeTypeConditional;
        cp.conditional.handle = G->handle;
        cp.conditional.type = cudaGraphCondTypeWhile;
        cp.conditional.size = 1;
        cudaGraphNode_t cnode;
        VEMG_CHECK_CUDA(cudaGraphAddNode(&cnode, G->g, frontier.data(), nullptr, frontier.size(), &cp));
        cudaGraph_t body = cp.conditional.phGraph_out[0];
        count = 0;
        VEMG_CHECK_CUDA(cudaStreamBeginCaptureToGraph(cs, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
        bphase_direction(h, W, cs);
        bphase_step(h, W, cs, G->handle, 1);
        VEMG_CHECK_CUDA(cudaStreamEndCapture(cs, &body));
        G->k_body = count;
        count = 0;
        VEMG_CHECK_CUDA(cudaStreamBeginCaptureToGraph(cs, G->g, &cnode, nullptr, 1, cudaStreamCaptureModeThreadLocal));
        bphase_post(h, W, cs);
        captured = G->g;
        VEMG_CHECK_CUDA(cudaStreamEndCapture(cs, &captured));
        G->k_post = count;
        VEMG_CHECK_CUDA(cudaGraphInstantiate(&G->exec, G->g, 0));
    } catch (...) {
        cudaStreamDestroy(cs);
        b_count = saved;
        release_batch_graphs(W);
        throw;
    }
    b_count = saved;
    VEMG_CHECK_CUDA(cudaStreamDestroy(cs));
}

void release_batch(vemg_hierarchy *h) {
    BatchWork *W = h->batch;
    if (!W) return;
    release_batch_graphs(W);
    W->arena.release();
    delete W;
    h->batch = nullptr;
}

__global__ void k_to_f32(int64_t n, const double *__restrict__ a, float *__restrict__ b) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) b[i] = (float)a[i];
}

__global__ void k_recip(int n, const double *__restrict__ d, void *out, int fp32) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double v = 1.0 / d[i];
    if (fp32) ((float *)out)[i] = (float)v;
    else ((double *)out)[i] = v;
}

static const void *values(Arena &ar, const double *v, int64_t n, bool fp32, cudaStream_t s) {
    if (!fp32) return v;
    float *f = ar.alloc<float>(n);
    if (n > 0) {
        k_to_f32<<<grid_for(n, 256), 256, 0, s>>>(n, v, f);
        VEMG_CHECK_LAUNCH();
    }
    return f;
}

// A chain operator's copy (BRows). colour: a level's matrix, its diagonal left out and the entries of
// earlier colours first.
__global__ void k_brows_fill(int n, const int *__restrict__ rp, const int *__restrict__ ci, const double *__restrict__ v,
                             const int *__restrict__ colour, int2 *ent, int *oci, double *ov, int *lo) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const int c0 = colour ? colour[r] : 0;
    int64_t o = (int64_t)rp[r] - (colour ? r : 0);
    for (int pass = colour ? 0 : 1; pass < 2; ++pass) {
        for (int k = rp[r]; k < rp[r + 1]; ++k) {
            const int j = ci[k];
            if (colour && (j == r || (colour[j] < c0) != (pass == 0))) continue;
            if (ent) {
                ent[o] = make_int2(j, __float_as_int((float)v[k]));
            } else {
                oci[o] = j;
                ov[o] = v[k];
            }
            ++o;
        }
        if (pass == 0) lo[r] = (int)(o - ((int64_t)rp[r] - r));
    }
}

__global__ void k_brows_info(int n, const int *__restrict__ crow, const int *__restrict__ rp, const int *__restrict__ lo,
                             int4 *info) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int r = crow[i];
    info[i] = make_int4(r, rp[r] - r, lo[r], rp[r + 1] - rp[r] - 1);
}

// Parts a row is split into: where the rows of one launch do not fill a quarter of the chip (152 SMs x 2048
// threads; half or an eighth of it measured 2 to 5% slower), a launch lasts as long as a row's chain of loads, which parts of about four entries cut. A
// warp must hold a row's parts at every launch shape, up to 32 lanes a row; the lanes that the widest
// loads would take count here, so that the parts (and with them the sums' order) do not depend on the
// shape.
static int parts_shift(int K, bool fp32, double rows, double mean) {
    const double lanes = std::max(1, K / (fp32 ? 4 : 2));
    int qsh = 0;
    while (std::min(K, 32) << (qsh + 1) <= 32 && mean > 4.0 * (1 << qsh) && rows * lanes * (2 << qsh) <= 152.0 * 512.0)
        ++qsh;
    return qsh;
}

static BRows outer_rows(const DCsr &A, const void *v) {
    BRows R;
    R.rp = A.rp;
    R.ci = A.ci;
    R.v = v;
    return R;
}

static BRows chain_rows(Arena &ar, const DCsr &A, const int *colour, const int *crow, double rows, int K, bool fp32, cudaStream_t s) {
    BRows R;
    const int64_t nnz = (int64_t)A.nnz - (colour ? A.n : 0);
    R.rp = A.rp;
    R.diag = colour != nullptr;
    R.qsh = parts_shift(K, fp32, rows, (double)nnz / std::max(A.n, 1));
    if (!fp32 && !colour) {   // as the setup keeps it: copies would take some 110 bytes a node
        R.ci = A.ci;
        R.v = A.v;
        return R;
    }
    int2 *ent = fp32 ? ar.alloc<int2>(nnz) : nullptr;
    int *ci = fp32 ? nullptr : ar.alloc<int>(nnz), *lo = colour ? ar.alloc<int>(A.n) : nullptr;
    double *v = fp32 ? nullptr : ar.alloc<double>(nnz);
    if (A.n > 0) {
        k_brows_fill<<<grid_for(A.n, 128), 128, 0, s>>>(A.n, A.rp, A.ci, A.v, colour, ent, ci, v, lo);
        VEMG_CHECK_LAUNCH();
    }
    R.ent = ent;
    R.ci = ci;
    R.v = v;
    R.lo = lo;
    if (colour) {
        int4 *info = ar.alloc<int4>(A.n);
        if (A.n > 0) {
            k_brows_info<<<grid_for(A.n, 256), 256, 0, s>>>(A.n, crow, A.rp, lo, info);
            VEMG_CHECK_LAUNCH();
        }
        R.info = info;
    }
    return R;
}

static BChain *build_bchain(const Chain &C, int K, bool fp32, Arena &ar, cudaStream_t s) {
    BChain *B = new BChain();
    try {
        B->nlev = C.nlev;
        B->direct = C.direct;
        B->nc = C.nc;
        B->G = C.G;
        if (C.direct && fp32) B->Gf = (const float *)values(ar, C.G, (int64_t)C.nc * C.nc, true, s);
        for (int l = 0; l < C.nlev; ++l) {
            const Level &L = C.lv[l];
            BLevel &T = B->lv[l];
            T.n = L.A.n;
            T.ncolours = L.ncolours;
            T.cptr = L.cptr;
            T.A = chain_rows(ar, L.A, L.colour, L.crow, (double)L.A.n / std::max(L.ncolours, 1), K, fp32, s);
            void *di = fp32 ? (void *)ar.alloc<float>(L.A.n) : (void *)ar.alloc<double>(L.A.n);
            k_recip<<<grid_for(L.A.n, 256), 256, 0, s>>>(L.A.n, L.diag, di, fp32);
            VEMG_CHECK_LAUNCH();
            T.dinv = di;
            if (l + 1 < C.nlev) {
                T.P = chain_rows(ar, L.P, nullptr, nullptr, L.A.n, K, fp32, s);
                T.PT = chain_rows(ar, L.PT, nullptr, nullptr, C.lv[l + 1].A.n, K, fp32, s);
            }
        }
    } catch (...) {
        delete B;
        throw;
    }
    return B;
}

BatchWork *new_batch_work(vemg_hierarchy *h, int K, cudaStream_t s);

static BatchWork *batch_work(vemg_hierarchy *h, int K, cudaStream_t s) {
    if (h->batch && h->batch->K == K) return h->batch;
    VEMG_CHECK_CUDA(cudaStreamSynchronize(s));
    release_batch(h);
    h->batch = new_batch_work(h, K, s);
    return h->batch;
}

// The autotuner: for each class of row kernel, every candidate shape (lanes per row 4, 8, 16, 32
// up to K; 2, 4 or 8 warps per block) is launched on a representative operation of this
// hierarchy at this batch width (class 0: the largest colour of the finest A_bar level swept
// over all its entries; class 1: the residual of that level; class 2: the outer q = A p), one
// warm-up and two timed launches each (CUDA events), and the fastest shape is kept. The vectors
// are the batch's own work buffers (zeroed); the per-column arithmetic does not depend on the shape.
template <class XT>
static void autotune_t(vemg_hierarchy *h, BatchWork *W, cudaStream_t s) {
    const int K = W->K;
    const BLevel &L = W->bbar->lv[0];
    XT *lx = (XT *)W->lx[1][0], *lb = (XT *)W->lb[1][0], *lr = (XT *)W->lr[1][0];
    const size_t vb = sizeof(XT) * (size_t)L.n * K;
    VEMG_CHECK_CUDA(cudaMemsetAsync(lx, 0, vb, s));
    VEMG_CHECK_CUDA(cudaMemsetAsync(lb, 0, vb, s));
    VEMG_CHECK_CUDA(cudaMemsetAsync(W->P, 0, sizeof(double) * (size_t)h->nu * K, s));
    int cbig = 0;
    for (int c = 1; c < L.ncolours; ++c)
        if (L.cptr[c + 1] - L.cptr[c] > L.cptr[cbig + 1] - L.cptr[cbig]) cbig = c;
    cudaEvent_t e0, e1;
    VEMG_CHECK_CUDA(cudaEventCreate(&e0));
    VEMG_CHECK_CUDA(cudaEventCreate(&e1));
    int64_t *saved = b_count;
    b_count = nullptr;
    try {
        for (int cls = 0; cls < 3; ++cls) {
            float best = 0.f;
            for (int kw : {4, 8, 16, 32}) {
                if (kw > K) continue;
                for (int wp : {2, 4, 8}) {
                    auto run = [&]() {
                        if (cls == 0)
                            brow<BOP_SOR, packed<XT>(), XT, XT, XT, XT, XT>(
                                L.A, L.cptr[cbig + 1] - L.cptr[cbig], L.A.info + L.cptr[cbig], ROW_ALL,
                                (const XT *)L.dinv, lb, lx, lx, K, -1, s, 0, kw, wp);
                        else if (cls == 1)
                            brow<BOP_UPPER, packed<XT>(), XT, XT, XT, XT, XT>(L.A, L.n, nullptr, ROW_UPPER,
                                                                             (const XT *)nullptr, lb, lx, lr, K, -1,
                                                                             s, 1, kw, wp);
                        else
                            brow<BOP_SPMV, false, double, double, double, double, double>(
                                W->Aout, h->nu, nullptr, ROW_ALL, (const double *)nullptr, (const double *)nullptr,
                                W->P, W->Q, K, -1, s, 2, kw, wp);
                    };
                    run();
                    VEMG_CHECK_CUDA(cudaEventRecord(e0, s));
                    run();
                    run();
                    VEMG_CHECK_CUDA(cudaEventRecord(e1, s));
                    VEMG_CHECK_CUDA(cudaEventSynchronize(e1));
                    float ms = 0.f;
                    VEMG_CHECK_CUDA(cudaEventElapsedTime(&ms, e0, e1));
                    const float us = 500.f * ms;   // per launch
                    W->tune.tried++;
                    if (W->tune.kw[cls] == 0 || us < best) {
                        best = us;
                        W->tune.kw[cls] = kw;
                        W->tune.warps[cls] = wp;
                        W->tune.us[cls] = us;
                    }
                }
            }
        }
    } catch (...) {
        b_count = saved;
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
        throw;
    }
    b_count = saved;
    VEMG_CHECK_CUDA(cudaEventDestroy(e0));
    VEMG_CHECK_CUDA(cudaEventDestroy(e1));
}

static void autotune(vemg_hierarchy *h, BatchWork *W, cudaStream_t s) {
    if (W->K < 4) return;   // one lane per row and column: no shape to choose
    if (h->precision != VEMG_PREC_FP64) autotune_t<float>(h, W, s);
    else autotune_t<double>(h, W, s);
}

static void fill_batch_work(vemg_hierarchy *h, BatchWork *W, cudaStream_t s) {
    const int K = W->K;
    Arena &ar = W->arena;
    int64_t N = (int64_t)h->n * K;
    W->X = ar.alloc<double>(N);
    W->R = ar.alloc<double>(N);
    W->Z = ar.alloc<double>(N);
    W->P = ar.alloc<double>(N);
    W->Q = ar.alloc<double>(N);
    W->B = ar.alloc<double>(N);
    VEMG_CHECK_CUDA(cudaMemsetAsync(W->Q, 0, sizeof(double) * N, s));
    VEMG_CHECK_CUDA(cudaMemsetAsync(W->Z, 0, sizeof(double) * N, s));
    const bool fp32 = h->precision != VEMG_PREC_FP64;
    size_t es = fp32 ? sizeof(float) : sizeof(double);
    const Chain *chains[2] = {&h->surf, single_chain(h) ? &the_chain(h) : &h->bar};
    if (!single_chain(h)) W->bsurf = build_bchain(h->surf, K, fp32, ar, s);
    W->bbar = build_bchain(*chains[1], K, fp32, ar, s);
    if (h->bc == VEMG_NEUMANN) {
        W->Aout = outer_rows(h->A, h->A.v);
        W->caller_of = h->new2old;
    } else {
        const DCsr &A0 = h->bar.lv[0].A;
        W->Aout = outer_rows(A0, A0.v);
        W->caller_of = h->new2old + h->mtop;
    }
    for (int ch = 0; ch < 2; ++ch)
        for (int l = 0; l < chains[ch]->nlev && (ch == 1 || !single_chain(h)); ++l) {
            int64_t m = (int64_t)chains[ch]->lv[l].A.n * K;
            W->lx[ch][l] = ar.alloc<char>((int64_t)es * m);
            W->lb[ch][l] = ar.alloc<char>((int64_t)es * m);
            W->lr[ch][l] = ar.alloc<char>((int64_t)es * m);
        }
    if (!single_chain(h)) {
        W->ET = outer_rows(h->ET, h->ET.v);
        W->E = outer_rows(h->E, values(ar, h->E.v, h->E.nnz, fp32, s));
        if (fp32) W->Rb32 = ar.alloc<float>((int64_t)(h->n - h->mtop) * K);
    }
    W->sc = ar.alloc<double>(B_COUNT * K + G_COUNT);
    W->part = ar.alloc<double>((int64_t)5 * stage1_blocks(N) * K);
    W->ctr = ar.alloc<unsigned>(2);
    VEMG_CHECK_CUDA(cudaMemsetAsync(W->ctr, 0, sizeof(unsigned) * 2, s));
    VEMG_CHECK_CUDA(cudaStreamSynchronize(s));
    autotune(h, W, s);
    VEMG_CHECK_CUDA(cudaStreamSynchronize(s));
}

BatchWork *new_batch_work(vemg_hierarchy *h, int K, cudaStream_t s) {
    BatchWork *W = new BatchWork();
    W->K = K;
    try {
        fill_batch_work(h, W, s);
    } catch (...) {
        cudaStreamSynchronize(s);   // what was enqueued on the arrays
        W->arena.release();
        delete W;
        throw;
    }
    return W;
}

int solve_batch(vemg_hierarchy *h, int k, const double *Bin, int64_t ldb, double *Xout, int64_t ldx, double rtol,
                int max_it, vemg_info *infos, cudaStream_t s) {
    if (k == 0) return VEMG_OK;
    if (k > kMaxK || h->precond == VEMG_PRECOND_NONE) throw Error{VEMG_EINVAL};
    prepare_solve(h, s);
    int K = 1;
    while (K < k) K *= 2;
    BatchWork *W = batch_work(h, K, s);
    TuneScope tune(&W->tune);
    b_count = &h->launches;
    const int nu = h->nu;
    k_binit<<<1, 1, 0, s>>>(W->sc, K, rtol, max_it);
    BATCH_LAUNCHED();
    const unsigned tiles = (unsigned)((nu + kTile - 1) / kTile), across = (unsigned)((K + kTile - 1) / kTile);
    k_bgather<<<dim3(tiles, across), 256, 0, s>>>(nu, K, k, ldb, W->caller_of, Bin, W->B);
    BATCH_LAUNCHED();
    // with a probe on, the same phases are launched on the stream (profilers see every kernel)
    const bool use_graph = h->probe.kind == PROBE_NONE;
    if (!W->graphs) build_batch_graphs(h, W);
    BatchGraphs *G = W->graphs;
    if (use_graph) {
        VEMG_CHECK_CUDA(cudaGraphLaunch(G->exec, s));   // the whole batched solve, one launch
    } else {
        bphase_pre(h, W, s);
        for (;;) {
            double cont = 0.0;
            VEMG_CHECK_CUDA(cudaMemcpyAsync(&cont, gsc(W) + G_CONT, sizeof(double), cudaMemcpyDeviceToHost, s));
            VEMG_CHECK_CUDA(cudaStreamSynchronize(s));
            if (cont == 0.0) break;
            bphase_direction(h, W, s);
            bphase_step(h, W, s, 0, 0);
        }
        bphase_post(h, W, s);
    }
    std::vector<double> hs(B_COUNT * K + G_COUNT);
    VEMG_CHECK_CUDA(cudaMemcpyAsync(hs.data(), W->sc, sizeof(double) * hs.size(), cudaMemcpyDeviceToHost, s));
    int ntop = h->bc == VEMG_DIRICHLET_TOP ? h->mtop : 0;
    k_bscatter<<<dim3(tiles, across), 256, 0, s>>>(nu, K, k, ldx, W->caller_of, W->X, Xout);
    BATCH_LAUNCHED();
    if (ntop > 0) {
        k_btops<<<grid_for((int64_t)ntop * k, 256), 256, 0, s>>>(ntop, k, ldx, h->tops, Xout);
        BATCH_LAUNCHED();
    }
    VEMG_CHECK_CUDA(cudaStreamSynchronize(s));
    int rounds = (int)hs[B_COUNT * K + G_ITERS];
    if (use_graph) h->launches += G->k_pre + G->k_post + (int64_t)rounds * G->k_body;
    int rc = VEMG_OK;
    for (int c = 0; c < k; ++c) {
        vemg_info &in = infos[c];
        double bn = hs[B_BN * K + c];
        in.iters = (int)hs[B_ITERS * K + c];
        in.relres = bn > 0.0 ? hs[B_RN * K + c] / bn : 0.0;
        in.true_relres = bn > 0.0 ? hs[B_TRUE * K + c] / bn : 0.0;
        in.b_mean = hs[B_BMEAN * K + c];
        if (hs[B_ZERO * K + c] != 0.0) in.status = VEMG_OK;
        else if (hs[B_FLAG * K + c] != 0.0) in.status = VEMG_EBREAKDOWN;
        else if (hs[B_CONV * K + c] != 0.0) in.status = VEMG_OK;
        else in.status = VEMG_ENOTCONV;
        if (in.status != VEMG_OK && rc == VEMG_OK) rc = in.status;
    }
    return rc;
}

}  // namespace vemg

// ------------------------------------------------------------------------------------------
// continuous batching: an engine holds K column slots of one hierarchy. A request is admitted into
// a free slot between iterations (its column is prepared and marked fresh, so its first direction
// is p = z - mu while the other columns continue their own recurrences); every step advances all
// occupied slots by whole iterations; a finished slot is retired (x copied out) and reused.

namespace vemg {

struct Engine {
    vemg_hierarchy *h = nullptr;
    BatchWork *W = nullptr;
    cudaStream_t s = nullptr;
    cudaGraphExec_t step = nullptr;
    cudaGraph_t gstep = nullptr;
    int64_t k_step = 0;
    std::vector<int> used;        // slot occupied
    double *hsc = nullptr;        // pinned copy of the per-column scalars
    double *colpart = nullptr;    // single-column reduction partials
    int ncolblk = 0;
};

static constexpr int kColBlocks = 128;

// sum over rows of column c of a (or of a^2; with p: of a + alpha p); per-block partials
__global__ void k_col_sum(int n, int K, int c, const double *__restrict__ a, int square, double *part,
                          const double *__restrict__ p = nullptr, const double *__restrict__ sc = nullptr) {
    __shared__ double sh[256];
    double v = 0.0;
    const double alpha = p ? sc[B_ALPHA * K + c] : 0.0;
    for (int i = blockIdx.x * 256 + threadIdx.x; i < n; i += kColBlocks * 256) {
        double x = a[(int64_t)i * K + c];
        if (p) x = fma(alpha, p[(int64_t)i * K + c], x);
        v += square ? x * x : x;
    }
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

// admission of column c: after the sum of b (mode 0) or of the projected b squared (mode 1)
__global__ void k_col_admit(int mode, int neumann, double inv_n, int K, int c, const double *__restrict__ part,
                            double *sc, double tol, int maxit) {
    double t = 0.0;
    for (int k = 0; k < kColBlocks; ++k) t += part[k];
    if (mode == 0) {
        sc[B_BMEAN * K + c] = neumann ? t * inv_n : 0.0;
        return;
    }
    double bn = sqrt(t);
    for (int slot = 0; slot < B_COUNT; ++slot)
        if (slot != B_BMEAN) sc[slot * K + c] = 0.0;
    sc[B_BN * K + c] = bn;
    sc[B_TOL * K + c] = tol;
    sc[B_MAXIT * K + c] = (double)maxit;
    sc[B_FRESH * K + c] = 1.0;
    if (bn == 0.0) {
        sc[B_ZERO * K + c] = 1.0;
        sc[B_CONV * K + c] = 1.0;
    }
}

__global__ void k_col_gather(int nu, int K, int c, const int *__restrict__ caller_of, const double *__restrict__ b,
                             double *__restrict__ B) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < nu) B[(int64_t)i * K + c] = b[caller_of[i]];
}

// b -= mean, r = b, x = p = z = q = 0 in column c
__global__ void k_col_prepare(int nu, int K, int c, const double *__restrict__ sc, double *B, double *R, double *X,
                              double *P, double *Z, double *Q, float *rb32, int64_t off32) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nu) return;
    int64_t e = (int64_t)i * K + c;
    double bi = B[e] - sc[B_BMEAN * K + c];
    B[e] = bi;
    R[e] = bi;
    if (rb32 && e >= off32) rb32[e - off32] = (float)bi;
    X[e] = 0.0;
    P[e] = 0.0;
    Z[e] = 0.0;
    Q[e] = 0.0;
}

__global__ void k_col_mean(int K, int c, const double *__restrict__ part, double inv_n, double *sc) {
    double t = 0.0;
    for (int k = 0; k < kColBlocks; ++k) t += part[k];
    sc[B_XMEAN * K + c] = t * inv_n;
}

// x = X + alpha P - mean of column c in the caller's order
__global__ void k_col_scatter(int nu, int K, int c, int neumann, const int *__restrict__ caller_of,
                              const int *__restrict__ tops, int ntop, const double *__restrict__ sc,
                              const double *__restrict__ X, const double *__restrict__ P, double *__restrict__ x) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    const double mu = neumann ? sc[B_XMEAN * K + c] : 0.0, alpha = sc[B_ALPHA * K + c];
    if (i < nu) x[caller_of[i]] = fma(alpha, P[(int64_t)i * K + c], X[(int64_t)i * K + c]) - mu;
    if (i < ntop) x[tops[i]] = 0.0;
}

// a retired slot is frozen (zero right-hand side, converged) until it is admitted again
__global__ void k_col_free(int nu, int K, int c, double *sc, double *B, double *R, double *X, double *P, float *rb32,
                           int64_t off32) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < nu) {
        int64_t e = (int64_t)i * K + c;
        B[e] = 0.0;
        R[e] = 0.0;
        if (rb32 && e >= off32) rb32[e - off32] = 0.0f;
        X[e] = 0.0;
        P[e] = 0.0;
    }
    if (i == 0) {
        for (int slot = 0; slot < B_COUNT; ++slot) sc[slot * K + c] = 0.0;
        sc[B_ZERO * K + c] = 1.0;
        sc[B_CONV * K + c] = 1.0;
    }
}

__global__ void k_engine_init(double *sc, int K) {
    for (int i = 0; i < B_COUNT * K + G_COUNT; ++i) sc[i] = 0.0;
    for (int c = 0; c < K; ++c) {
        sc[B_ZERO * K + c] = 1.0;
        sc[B_CONV * K + c] = 1.0;
    }
}

BatchWork *new_batch_work(vemg_hierarchy *h, int K, cudaStream_t s);

}  // namespace vemg

using namespace vemg;

struct vemg_engine : vemg::Engine {};

extern "C" {

int vemg_engine_create(vemg_hierarchy *h, int slots, void *stream, vemg_engine **out) {
    if (!h || !out || slots < 1 || slots > kMaxK || h->precond == VEMG_PRECOND_NONE) return VEMG_EINVAL;
    *out = nullptr;
    vemg_engine *e = new vemg_engine();
    try {
        cudaStream_t s = (cudaStream_t)stream;
        prepare_solve(h, s);
        int K = 1;
        while (K < slots) K *= 2;
        e->h = h;
        e->s = s;
        e->W = new_batch_work(h, K, s);
        e->used.assign(K, 0);
        VEMG_CHECK_CUDA(cudaMallocHost(&e->hsc, sizeof(double) * (B_COUNT * K + G_COUNT)));
        e->colpart = e->W->arena.alloc<double>(kColBlocks);
        k_engine_init<<<1, 1, 0, s>>>(e->W->sc, K);
        VEMG_CHECK_LAUNCH();
        // one iteration of every occupied column, as a graph
        TuneScope tune(&e->W->tune);
        cudaStream_t cs;
        VEMG_CHECK_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
        int64_t count = 0;
        b_count = &count;
        VEMG_CHECK_CUDA(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
        bphase_direction(h, e->W, cs);
        bphase_step(h, e->W, cs, 0, 0);
        VEMG_CHECK_CUDA(cudaStreamEndCapture(cs, &e->gstep));
        b_count = nullptr;
        e->k_step = count;
        VEMG_CHECK_CUDA(cudaStreamDestroy(cs));
        VEMG_CHECK_CUDA(cudaGraphInstantiate(&e->step, e->gstep, 0));
        VEMG_CHECK_CUDA(cudaStreamSynchronize(s));
    } catch (const Error &err) {
        b_count = nullptr;
        vemg_engine_destroy(e);
        return err.code;
    } catch (...) {
        b_count = nullptr;
        vemg_engine_destroy(e);
        return VEMG_EINTERNAL;
    }
    *out = e;
    return VEMG_OK;
}

void vemg_engine_destroy(vemg_engine *e) {
    if (!e) return;
    if (e->s) cudaStreamSynchronize(e->s);
    if (e->step) cudaGraphExecDestroy(e->step);
    if (e->gstep) cudaGraphDestroy(e->gstep);
    if (e->hsc) cudaFreeHost(e->hsc);
    if (e->W) {
        e->W->arena.release();
        delete e->W;
    }
    delete e;
}

int vemg_engine_admit(vemg_engine *e, const double *b_dev, double rtol, int max_it, int *slot) {
    if (!e || !b_dev || !slot || !(rtol >= 0.0) || max_it < 0) return VEMG_EINVAL;
    int c = -1;
    for (int k = 0; k < (int)e->used.size(); ++k)
        if (!e->used[k]) {
            c = k;
            break;
        }
    if (c < 0) return VEMG_ENOMEM;
    try {
        vemg_hierarchy *h = e->h;
        BatchWork *W = e->W;
        const int nu = h->nu, K = W->K;
        const bool neu = h->bc == VEMG_NEUMANN;
        cudaStream_t s = e->s;
        k_col_gather<<<grid_for(nu, 256), 256, 0, s>>>(nu, K, c, W->caller_of, b_dev, W->B);
        VEMG_CHECK_LAUNCH();
        k_col_sum<<<kColBlocks, 256, 0, s>>>(nu, K, c, W->B, 0, e->colpart);
        VEMG_CHECK_LAUNCH();
        k_col_admit<<<1, 1, 0, s>>>(0, neu, 1.0 / nu, K, c, e->colpart, W->sc, rtol, max_it);
        VEMG_CHECK_LAUNCH();
        k_col_prepare<<<grid_for(nu, 256), 256, 0, s>>>(nu, K, c, W->sc, W->B, W->R, W->X, W->P, W->Z, W->Q, W->Rb32,
                                                        rb32_offset(h, W));
        VEMG_CHECK_LAUNCH();
        k_col_sum<<<kColBlocks, 256, 0, s>>>(nu, K, c, W->B, 1, e->colpart);
        VEMG_CHECK_LAUNCH();
        k_col_admit<<<1, 1, 0, s>>>(1, neu, 1.0 / nu, K, c, e->colpart, W->sc, rtol, max_it);
        VEMG_CHECK_LAUNCH();
        h->launches += 6;
    } catch (const Error &err) {
        return err.code;
    }
    e->used[c] = 1;
    *slot = c;
    return VEMG_OK;
}

int vemg_engine_launch(vemg_engine *e, int iters) {
    if (!e || iters < 0) return VEMG_EINVAL;
    for (int k = 0; k < iters; ++k) {
        cudaError_t err = cudaGraphLaunch(e->step, e->s);
        if (err != cudaSuccess) {
            set_last_cuda_error(err, "cudaGraphLaunch", __FILE__, __LINE__);
            return VEMG_ECUDA;
        }
    }
    e->h->launches += (int64_t)iters * e->k_step;
    const int K = e->W->K;
    cudaError_t err = cudaMemcpyAsync(e->hsc, e->W->sc, sizeof(double) * (B_COUNT * K + G_COUNT),
                                      cudaMemcpyDeviceToHost, e->s);
    if (err != cudaSuccess) {
        set_last_cuda_error(err, "cudaMemcpyAsync", __FILE__, __LINE__);
        return VEMG_ECUDA;
    }
    return VEMG_OK;
}

int vemg_engine_wait(vemg_engine *e) {
    if (!e) return VEMG_EINVAL;
    cudaError_t err = cudaStreamSynchronize(e->s);
    if (err != cudaSuccess) {
        set_last_cuda_error(err, "cudaStreamSynchronize", __FILE__, __LINE__);
        return VEMG_ECUDA;
    }
    return VEMG_OK;
}

int vemg_engine_query(const vemg_engine *e, int *busy) {
    if (!e || !busy) return VEMG_EINVAL;
    cudaError_t err = cudaStreamQuery(e->s);
    if (err == cudaErrorNotReady) {
        *busy = 1;
        return VEMG_OK;
    }
    if (err != cudaSuccess) {
        set_last_cuda_error(err, "cudaStreamQuery", __FILE__, __LINE__);
        return VEMG_ECUDA;
    }
    *busy = 0;
    return VEMG_OK;
}

int vemg_engine_poll(const vemg_engine *e, int slot, vemg_info *info, int *state) {
    if (!e || !state || slot < 0 || slot >= (int)e->used.size()) return VEMG_EINVAL;
    if (!e->used[slot]) {
        *state = VEMG_SLOT_FREE;
        return VEMG_OK;
    }
    const int K = e->W->K;
    const double *sc = e->hsc;
    bool conv = sc[B_CONV * K + slot] != 0.0, flag = sc[B_FLAG * K + slot] != 0.0;
    bool out = sc[B_ITERS * K + slot] >= sc[B_MAXIT * K + slot] || sc[B_STALL * K + slot] != 0.0;
    *state = (conv || flag || out) ? VEMG_SLOT_DONE : VEMG_SLOT_RUNNING;
    if (info) {
        double bn = sc[B_BN * K + slot];
        info->iters = (int)sc[B_ITERS * K + slot];
        info->relres = bn > 0.0 ? sc[B_RN * K + slot] / bn : 0.0;
        info->true_relres = -1.0;
        info->b_mean = sc[B_BMEAN * K + slot];
        info->status = sc[B_ZERO * K + slot] != 0.0 ? VEMG_OK
                       : flag                       ? VEMG_EBREAKDOWN
                       : conv                       ? VEMG_OK
                                                    : VEMG_ENOTCONV;
    }
    return VEMG_OK;
}

int vemg_engine_retire(vemg_engine *e, int slot, double *x_dev) {
    if (!e || !x_dev || slot < 0 || slot >= (int)e->used.size() || !e->used[slot]) return VEMG_EINVAL;
    try {
        vemg_hierarchy *h = e->h;
        BatchWork *W = e->W;
        const int nu = h->nu, K = W->K;
        const bool neu = h->bc == VEMG_NEUMANN;
        cudaStream_t s = e->s;
        if (neu) {
            k_col_sum<<<kColBlocks, 256, 0, s>>>(nu, K, slot, W->X, 0, e->colpart, W->P, W->sc);
            VEMG_CHECK_LAUNCH();
            k_col_mean<<<1, 1, 0, s>>>(K, slot, e->colpart, 1.0 / nu, W->sc);
            VEMG_CHECK_LAUNCH();
        }
        int ntop = neu ? 0 : h->mtop;
        k_col_scatter<<<grid_for(std::max(nu, ntop), 256), 256, 0, s>>>(nu, K, slot, neu, W->caller_of, h->tops, ntop,
                                                                         W->sc, W->X, W->P, x_dev);
        VEMG_CHECK_LAUNCH();
        k_col_free<<<grid_for(nu, 256), 256, 0, s>>>(nu, K, slot, W->sc, W->B, W->R, W->X, W->P, W->Rb32,
                                                     rb32_offset(h, W));
        VEMG_CHECK_LAUNCH();
        VEMG_CHECK_CUDA(cudaStreamSynchronize(s));
        h->launches += neu ? 4 : 2;
    } catch (const Error &err) {
        return err.code;
    }
    e->used[slot] = 0;
    return VEMG_OK;
}

int vemg_batch_tuning(const vemg_hierarchy *h, int *K, int *kw, int *warps, float *us) {
    if (!h || !K || !kw || !warps || !us) return VEMG_EINVAL;
    if (!h->batch) return VEMG_EINVAL;
    const BTune &t = h->batch->tune;
    *K = h->batch->K;
    for (int c = 0; c < 3; ++c) {
        kw[c] = t.kw[c];
        warps[c] = t.warps[c];
        us[c] = t.us[c];
    }
    return VEMG_OK;
}

int vemg_batch_set_tuning(vemg_hierarchy *h, int K, const int *kw, const int *warps, void *stream) {
    if (!h || !kw || !warps || K < 1 || K > kMaxK || (K & (K - 1)) || h->precond == VEMG_PRECOND_NONE)
        return VEMG_EINVAL;
    for (int c = 0; c < 3; ++c)
        if (!(kw[c] == 4 || kw[c] == 8 || kw[c] == 16 || kw[c] == 32) || !(warps[c] == 2 || warps[c] == 4 ||
                                                                          warps[c] == 8))
            return VEMG_EINVAL;
    try {
        cudaStream_t s = (cudaStream_t)stream;
        prepare_solve(h, s);
        BatchWork *W = batch_work(h, K, s);
        for (int c = 0; c < 3; ++c) {
            W->tune.kw[c] = kw[c];
            W->tune.warps[c] = warps[c];
            W->tune.us[c] = 0.f;
        }
        release_batch_graphs(W);   // recaptured with the new shapes at the next solve
    } catch (const Error &err) {
        return err.code;
    } catch (...) {
        return VEMG_EINTERNAL;
    }
    return VEMG_OK;
}

int vemg_engine_slots(const vemg_engine *e, int *slots, int *free_slots) {
    if (!e || !slots || !free_slots) return VEMG_EINVAL;
    *slots = (int)e->used.size();
    int f = 0;
    for (int u : e->used) f += !u;
    *free_slots = f;
    return VEMG_OK;
}

int vemg_engine_bytes(const vemg_engine *e, size_t *bytes) {
    if (!e || !bytes) return VEMG_EINVAL;
    *bytes = e->W->arena.bytes;
    return VEMG_OK;
}

}  // extern "C"
