// dense.cu -- the dense inverse of a coarsest level (at most 1024 rows): blocked Cholesky
// D = L L^T, the inverse X of L by recursive doubling, G = X^T X, all in tiles of 32 x 32 over the
// whole chip.
//
// The factor L is the one of the column-by-column algorithm bit for bit: every element is reduced
// by its products in ascending column order, each product and each difference rounded on its own, and
// divided by the pivot's root. A coarsest operator's condition number reaches 1e7, so a factor rounded
// in another order would move the inverse by 1e-9; the inverse of a given L is good to the root of that.
//
// FP64 bounds it: about n^3 / 2 multiply-adds at two per cycle and SM (the FP64 rate of this GPU),
// under the chain of n / 32 diagonal tiles that each need the update before them (79 us a tile: a root,
// a division and a rank-one update per column). Measured: n = 580 2.7 ms, n = 240 0.8 ms; with one block
// factoring column by column and one thread per column of the inverse substituting through L, n = 240
// took 7.2 ms and n = 985 and 580 together (the 256 x 256 x 32 mesh) 269 ms.
#include <algorithm>

#include "internal.cuh"

namespace vemg {

static constexpr int kT = kDenseTile;        // tile edge
static constexpr int kDT = 256;              // threads per tile: 8 x 32, four elements each

// acc(4 elements of the thread's tile) += A B for tiles in shared memory
__device__ __forceinline__ void tile_mac(double (&acc)[4], const double (&a)[kT][kT + 1], const double (&b)[kT][kT + 1],
                                         int ty, int tx) {
#pragma unroll 8
    for (int k = 0; k < kT; ++k) {
        const double bv = b[k][tx];
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] = __fma_rn(a[ty + 8 * q][k], bv, acc[q]);
    }
}

__device__ __forceinline__ void tile_load(double (&a)[kT][kT + 1], const double *__restrict__ src, int ld, int ti, int tj,
                                          int ty, int tx) {
#pragma unroll
    for (int q = 0; q < 4; ++q) a[ty + 8 * q][tx] = src[(int64_t)(ti * kT + ty + 8 * q) * ld + tj * kT + tx];
}

// Step k of the factorisation: the diagonal tile's factor into X's diagonal tile (A_kk is only
// read), L_ik in place of the tiles A_ik below it. Every block factors the diagonal tile along with
// the tile that it owns, so that the panel needs no launch of its own: block 0 stores the diagonal
// tile, block b the tile in row k + b.
__global__ void __launch_bounds__(kDT) k_chol_panel(int np, int k, double *A, double *X, int *err) {
    __shared__ double a[2 * kT][kT + 1];   // rows 0..31: the diagonal tile, 32..63: the block's tile
    __shared__ double piv;
    const int t = threadIdx.x, ty = t / kT, tx = t % kT, ti = k + (int)blockIdx.x;
    const int rows = blockIdx.x > 0 ? 2 * kT : kT;
    for (int r = ty; r < rows; r += 8)
        a[r][tx] = A[(int64_t)((r < kT ? k * kT : ti * kT - kT) + r) * np + k * kT + tx];
    __syncthreads();
    for (int j = 0; j < kT; ++j) {
        if (t == 0) {
            double d = a[j][j];
            if (!(d > 0.0)) {
                atomicCAS(err, 0, VEMG_EBREAKDOWN);
                d = 1.0;
            }
            piv = __dsqrt_rn(d);
        }
        __syncthreads();
        if (t < rows && t > j) a[t][j] = __ddiv_rn(a[t][j], piv);
        if (t == rows) a[j][j] = piv;
        __syncthreads();
        const int c = tx;   // column c > j of the rows below it: c .. rows - 1
        if (c > j)
            for (int i = ty; i < rows; i += 8)
                if (i >= c) a[i][c] = __dsub_rn(a[i][c], __dmul_rn(a[i][j], a[c][j]));
        __syncthreads();
    }
    double *dst = blockIdx.x > 0 ? A : X;
    const int r0 = blockIdx.x > 0 ? kT : 0;
#pragma unroll
    for (int q = 0; q < 4; ++q)
        dst[(int64_t)(ti * kT + ty + 8 * q) * np + k * kT + tx] = a[r0 + ty + 8 * q][tx];
}

// A_ij -= L_ik L_jk^T for k < j <= i (one block per tile of the lower triangle)
__global__ void __launch_bounds__(kDT) k_chol_update(int np, int k, double *A) {
    const int i = k + 1 + (int)blockIdx.y, j = k + 1 + (int)blockIdx.x;
    if (j > i) return;
    __shared__ double a[kT][kT + 1], b[kT][kT + 1];
    const int ty = threadIdx.x / kT, tx = threadIdx.x % kT;
    tile_load(a, A, np, i, k, ty, tx);
    tile_load(b, A, np, j, k, ty, tx);
    double *c = A + (int64_t)(i * kT + ty) * np + j * kT + tx;
    double acc[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[q] = c[(int64_t)8 * q * np];
    __syncthreads();
#pragma unroll 8
    for (int m = 0; m < kT; ++m) {
        const double bv = b[tx][m];
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] = __dsub_rn(acc[q], __dmul_rn(a[ty + 8 * q][m], bv));
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) c[(int64_t)8 * q * np] = acc[q];
}

// X_kk := the inverse of the factor's diagonal tile (one block per tile): elimination of [L_kk | I]
__global__ void __launch_bounds__(kDT) k_tri_diag(int np, double *X) {
    __shared__ double a[kT][kT + 1], w[kT][kT + 1];
    const int t = threadIdx.x, ty = t / kT, tx = t % kT, k = blockIdx.x;
    tile_load(a, X, np, k, k, ty, tx);
#pragma unroll
    for (int q = 0; q < 4; ++q) w[ty + 8 * q][tx] = ty + 8 * q == tx ? 1.0 : 0.0;
    __syncthreads();
    for (int j = 0; j < kT; ++j) {
        if (t <= j) w[j][t] = __ddiv_rn(w[j][t], a[j][j]);
        __syncthreads();
        if (tx <= j)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int i = ty + 8 * q;
                if (i > j) w[i][tx] = __fma_rn(-a[i][j], w[j][tx], w[i][tx]);
            }
        __syncthreads();
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) X[(int64_t)(k * kT + ty + 8 * q) * np + k * kT + tx] = w[ty + 8 * q][tx];
}

// Recursive doubling of X = L^-1: with the inverses of the diagonal blocks of s tiles known, the
// block below the first of each pair is X_RC = -X_RR (L_RC X_CC). half 0: T_RC = L_RC X_CC; half 1:
// X_RC = -X_RR T_RC. One block per tile; x = tile column within C, y = tile row within R, z = pair.
__global__ void __launch_bounds__(kDT) k_tri_inverse(int np, int s, int half, const double *L, double *X, double *T) {
    const int c0 = (int)blockIdx.z * 2 * s, r0 = c0 + s;
    const int i = r0 + (int)blockIdx.y, j = c0 + (int)blockIdx.x;
    if (i >= np / kT) return;
    __shared__ double a[kT][kT + 1], b[kT][kT + 1];
    const int ty = threadIdx.x / kT, tx = threadIdx.x % kT;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    const int k0 = half == 0 ? j : r0, k1 = half == 0 ? r0 - 1 : i;   // the triangular factor's tiles
    for (int k = k0; k <= k1; ++k) {
        tile_load(a, half == 0 ? L : X, np, i, k, ty, tx);
        tile_load(b, half == 0 ? X : T, np, k, j, ty, tx);
        __syncthreads();
        tile_mac(acc, a, b, ty, tx);
        __syncthreads();
    }
    double *dst = half == 0 ? T : X;
#pragma unroll
    for (int q = 0; q < 4; ++q)
        dst[(int64_t)(i * kT + ty + 8 * q) * np + j * kT + tx] = half == 0 ? acc[q] : -acc[q];
}

// G = X^T X, the lower triangle's tiles and their mirror images (exactly symmetric)
__global__ void __launch_bounds__(kDT) k_tri_square(int n, int np, const double *X, double *G) {
    const int i = blockIdx.y, j = blockIdx.x;
    if (j > i) return;
    __shared__ double a[kT][kT + 1], b[kT][kT + 1];
    const int ty = threadIdx.x / kT, tx = threadIdx.x % kT;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    for (int k = i; k < np / kT; ++k) {
        tile_load(a, X, np, k, i, ty, tx);
        tile_load(b, X, np, k, j, ty, tx);
        __syncthreads();
#pragma unroll 8
        for (int m = 0; m < kT; ++m) {
            const double bv = b[m][tx];
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[q] = __fma_rn(a[m][ty + 8 * q], bv, acc[q]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int r = i * kT + ty + 8 * q, c = j * kT + tx;
        if (r >= n || c >= n || c > r) continue;
        G[(int64_t)r * n + c] = acc[q];
        G[(int64_t)c * n + r] = acc[q];
    }
}

// gv = G v (v null: the constants), one warp per row
__global__ void k_dense_times(int n, const double *__restrict__ G, const double *__restrict__ v, double *__restrict__ gv) {
    const int row = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (row >= n) return;
    double s = 0.0;
    for (int k = lane; k < n; k += 32) s = __fma_rn(G[(int64_t)row * n + k], v ? v[k] : 1.0, s);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) gv[row] = s;
}

// G := Q G Q, Q = I - v v^T / (v^T v) (G symmetric, gv = G v), one block per row. Every block adds up
// v^T v and v^T G v in the same order.
__global__ void __launch_bounds__(kDT) k_dense_project(int n, double *__restrict__ G, const double *__restrict__ v,
                                                       const double *__restrict__ gv) {
    __shared__ double sv[2][kDT / 32];
    const int t = threadIdx.x, i = blockIdx.x;
    double p[2] = {0.0, 0.0};
    for (int k = t; k < n; k += kDT) {
        const double vk = v ? v[k] : 1.0;
        p[0] = __fma_rn(vk, vk, p[0]);
        p[1] = __fma_rn(vk, gv[k], p[1]);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) p[q] += __shfl_xor_sync(0xffffffffu, p[q], o);
        if ((t & 31) == 0) sv[q][t >> 5] = p[q];
    }
    __syncthreads();
    double nn = 0.0, vgv = 0.0;
    for (int w = 0; w < kDT / 32; ++w) {
        nn += sv[0][w];
        vgv += sv[1][w];
    }
    const double vi = (v ? v[i] : 1.0) / nn, gi = gv[i] / nn, c = vgv / nn;
    for (int j = t; j < n; j += kDT) {
        const double vj = v ? v[j] : 1.0;
        G[(int64_t)i * n + j] += vi * (vj * c - gv[j]) - gi * vj;
    }
}

// D (np x np, np = dense_padded(n); the rows and columns past n are those of the identity) is
// overwritten by its factor; G (n x n) receives the inverse of the leading n x n block. A pivot that
// is not positive sets *err.
void dense_spd_inverse(int n, double *D, double *G, int *err, cudaStream_t s) {
    const int np = dense_padded(n), m = np / kT;
    Scratch<double> X((int64_t)np * np), T((int64_t)np * np);
    for (int k = 0; k < m; ++k) {
        k_chol_panel<<<m - k, kDT, 0, s>>>(np, k, D, X, err);
        VEMG_CHECK_LAUNCH();
        if (k + 1 < m) {
            k_chol_update<<<dim3(m - 1 - k, m - 1 - k), kDT, 0, s>>>(np, k, D);
            VEMG_CHECK_LAUNCH();
        }
    }
    k_tri_diag<<<m, kDT, 0, s>>>(np, X);
    VEMG_CHECK_LAUNCH();
    for (int b = 1; b < m; b *= 2) {
        const dim3 grid(b, b, (m - b + 2 * b - 1) / (2 * b));   // pairs whose second block has a tile
        for (int half = 0; half < 2; ++half) {
            k_tri_inverse<<<grid, kDT, 0, s>>>(np, b, half, D, X, T);
            VEMG_CHECK_LAUNCH();
        }
    }
    k_tri_square<<<dim3(m, m), kDT, 0, s>>>(n, np, X, G);
    VEMG_CHECK_LAUNCH();
}

// G := Q G Q on the complement of v (null: the constants)
void dense_project(int n, double *G, const double *v, cudaStream_t s) {
    Scratch<double> gv(n);
    k_dense_times<<<grid_for((int64_t)n * 32, 256), 256, 0, s>>>(n, G, v, gv);
    VEMG_CHECK_LAUNCH();
    k_dense_project<<<n, kDT, 0, s>>>(n, G, v, gv);
    VEMG_CHECK_LAUNCH();
}

}  // namespace vemg
