// layout.cu -- the solve-phase layout of the hierarchy.
//
// The setup builds every operator in the natural ordering of its level (the ordering the
// method's definitions use). The solve reorders each multigrid level colour by colour, so that
// one colour of a multicolour SOR sweep is a contiguous range of rows, and stores every operator
// of the solve as a sliced ELL matrix (one warp per slice, entries of a slice interleaved so that
// the 32 threads read consecutive words). The fine ordering of the outer
// Krylov vectors is [top nodes in the colour order of the surface level 0; non-top nodes in the
// colour order of A_bar's level 0], so that the A_bar branch of the preconditioner reads its
// right-hand side as the trailing part of r with no gather.
#include <algorithm>
#include <cstring>

#include <cuda_bf16.h>

#include "internal.cuh"

namespace vemg {

__global__ void k_inverse_perm(int n, const int *__restrict__ s2n, int *n2s) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) n2s[s2n[i]] = i;
}

// steps of each slice (one warp per slice) and the elements they take
__global__ void k_sell_width(int nslices, const int *__restrict__ row0, const int *__restrict__ nrow,
                             const int *__restrict__ s2n, const int *__restrict__ rp, int split, int lsh, int *width,
                             int *elements, int *longest) {
    const int s = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (s >= nslices) return;
    unsigned len = 0;
    if (lane < nrow[s]) {
        const int r = row0[s] + lane, i = s2n ? s2n[r] : r;
        len = (unsigned)max(rp[i + 1] - rp[i] - split, 0);
    }
    const int w = (int)__reduce_max_sync(0xffffffffu, len);
    if (lane != 0) return;
    width[s] = (w + (1 << lsh) - 1) >> lsh;
    elements[s] = 32 * width[s];
    if (w > 0xffff) atomicMax(longest, w);
}

template <class VT>
__global__ void k_sell_fill(int nslices, const int *__restrict__ row0, const int *__restrict__ nrow,
                            const int *__restrict__ off, const int *__restrict__ width, const int *__restrict__ s2n,
                            const int *__restrict__ n2s, const int *__restrict__ rp, const int *__restrict__ ci,
                            const double *__restrict__ v, int *col, VT *val, unsigned long long *cnt) {
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int s = (int)(t / 32), lane = (int)(t % 32);
    if (s >= nslices) return;
    int o = off[s] + lane, w = width[s];
    int k = 0;
    if (lane < nrow[s]) {
        int r = row0[s] + lane;
        int i = s2n ? s2n[r] : r;
        for (int e = rp[i]; e < rp[i + 1]; ++e) {
            int c = ci[e];
            col[o + 32 * k] = n2s ? n2s[c] : c;
            val[o + 32 * k] = (VT)v[e];
            ++k;
        }
    }
    const unsigned entries = __reduce_add_sync(0xffffffffu, (unsigned)k);
    if (lane == 0) atomicAdd(cnt + 1, (unsigned long long)entries);   // one group
    for (; k < w; ++k) {
        col[o + 32 * k] = 0;
        val[o + 32 * k] = (VT)0;
    }
}

// The chains' form (sell.cuh): the first thread of each row walks the row and deals its entries to
// the row's lanes. split: the diagonal apart, the entries of earlier colours first (columns below
// the row's own: a row has no entry in its own colour but the diagonal). Unused places hold zeros.
// cnt: entries per group of the rows (group of a slice: gcol), of earlier colours and all.
template <class VT>
__global__ void k_sell_deal(int nslices, int lsh, const int *__restrict__ row0, const int *__restrict__ nrow,
                            const int *__restrict__ off, const int *__restrict__ width, const int *__restrict__ s2n,
                            const int *__restrict__ n2s, const int *__restrict__ rp, const int *__restrict__ ci,
                            const double *__restrict__ v, int split, int *col, VT *val, VT *dinv, int4 *meta,
                            unsigned *rl, int rl_wide, const int *__restrict__ gcol, unsigned long long *cnt) {
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int s = (int)(t / 32), lane = (int)(t % 32);
    if (s >= nslices) return;
    const int rows = 32 >> lsh, L = 1 << lsh, o = off[s], w = width[s];
    if (lane == 0) meta[s] = make_int4(row0[s], nrow[s], o, w);
    for (int k = 0; k < w; ++k) {
        col[o + 32 * k + lane] = 0;
        val[o + 32 * k + lane] = (VT)0;
    }
    __syncwarp();
    unsigned nlow = 0, k = 0;
    if (lane < nrow[s] && lane < rows) {
        const int r = row0[s] + lane, i = s2n ? s2n[r] : r;
        for (int pass = split ? 0 : 1; pass < 2; ++pass) {
            for (int e = rp[i]; e < rp[i + 1]; ++e) {
                const int c = ci[e];
                if (split && c == i) {
                    dinv[r] = (VT)(1.0 / v[e]);
                    continue;
                }
                const int cs = n2s ? n2s[c] : c;
                if (split && (cs < r) != (pass == 0)) continue;
                const int at = o + 32 * (int)(k >> lsh) + (int)(k & (L - 1)) * rows + lane;
                col[at] = cs;
                val[at] = (VT)v[e];
                ++k;
            }
            if (pass == 0) nlow = k;
        }
        if (rl_wide) {
            rl[2 * (int64_t)r] = nlow;
            rl[2 * (int64_t)r + 1] = k;
        } else {
            rl[r] = nlow | k << 16;
        }
    }
    nlow = __reduce_add_sync(0xffffffffu, nlow);
    k = __reduce_add_sync(0xffffffffu, k);
    if (lane != 0) return;
    if (nlow) atomicAdd(cnt + 2 * gcol[s], (unsigned long long)nlow);
    atomicAdd(cnt + 2 * gcol[s] + 1, (unsigned long long)k);
}

// Lanes per row of a chain's operator, by the rows that one launch works on and their mean length.
// A row per thread reads 32 rows' entries in consecutive words and is the better form while the
// rows alone fill half the chip (152 SMs x 2048 threads); below that a launch lasts as long as its
// longest chain of loads, which more lanes per row cut: four entries each is as far as it pays. In FP64
// every step of a warp holds a scheduler for 64 cycles however few of its lanes have an entry, and so does
// every level of the tree that adds the lanes up, so lanes pay half as far (a 131 x 113 x 25 solve: 9.7 ms;
// 10.2 with 0.62 of the FP32 limit and with all of it, 9.97 and 10.68 with a quarter and an eighth).
static int lanes_shift(double rows, double mean, bool fp32) {
    const double most = 152.0 * (fp32 ? 1024.0 : 512.0);
    int lsh = 0;
    while (lsh < 5 && mean > 4.0 * (1 << lsh) && rows * (2 << lsh) <= most) ++lsh;
    return lsh;
}

// slice s of the groups (group g: slices gs[g] .. gs[g + 1], rows from gr[g])
__global__ void k_slices(int nslices, int ngroups, const int *__restrict__ gr, const int *__restrict__ gs, int rows,
                         int *row0, int *nrow, int *gcol) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= nslices) return;
    int lo = 0, hi = ngroups;   // the last group whose first slice is at most s (an empty group has none)
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (gs[mid] <= s) lo = mid;
        else hi = mid;
    }
    const int r = gr[lo] + (s - gs[lo]) * rows;
    row0[s] = r;
    nrow[s] = min(rows, gr[lo + 1] - r);
    gcol[s] = lo;
}

// Build the sliced ELL of the rows s2n[0..n) of the CSR matrix A (natural order), columns mapped
// through n2s (null: identity). groups: row boundaries (solve order) that slices do not straddle.
// dinv: a level's matrix, its inverse diagonal apart from the slices. lsh < 0: an outer operator's form;
// else a chain's, with 1 << lsh lanes per row.
static Sell build_sell(Arena &ar, const DCsr &A, int n, const int *s2n, const int *n2s, int ncols,
                       const std::vector<int> &groups, bool fp32, void **dinv, std::vector<int> *gslice,
                       cudaStream_t s, int lsh = -1, std::vector<int64_t> *low = nullptr,
                       std::vector<int64_t> *all = nullptr) {
    const bool split = dinv != nullptr;
    Sell S;
    S.n = n;
    S.m = ncols;
    S.fp32 = fp32;
    S.lsh = lsh < 0 ? 0 : lsh;
    const int rows = 32 >> S.lsh;
    const int ngroups = std::max((int)groups.size() - 1, 0);
    std::vector<int> table(2 * (size_t)(ngroups + 1), 0);   // first row, first slice of each group
    for (int g = 0; g <= ngroups && !groups.empty(); ++g) {
        table[g] = groups[g];
        if (g > 0) table[ngroups + 1 + g] = table[ngroups + g] + (groups[g] - groups[g - 1] + rows - 1) / rows;
    }
    if (gslice) gslice->assign(table.begin() + ngroups + 1, table.end());
    S.nslices = table.back();
    S.row0 = ar.alloc<int>(S.nslices);
    S.nrow = ar.alloc<int>(S.nslices);
    S.width = ar.alloc<int>(S.nslices);
    S.off = ar.alloc<int>(S.nslices + 1);
    int longest = 0, total = 0;
    Scratch<int> gtab((int64_t)table.size()), gcol(S.nslices);
    if (S.nslices) {
        Scratch<int> lg(1), w32(S.nslices);
        VEMG_CHECK_CUDA(cudaMemsetAsync(lg, 0, sizeof(int), s));
        VEMG_CHECK_CUDA(cudaMemcpyAsync(gtab, table.data(), sizeof(int) * table.size(), cudaMemcpyHostToDevice, s));
        k_slices<<<grid_for(S.nslices, 256), 256, 0, s>>>(S.nslices, ngroups, gtab, gtab.p + ngroups + 1, rows, S.row0,
                                                          S.nrow, gcol);
        VEMG_CHECK_LAUNCH();
        k_sell_width<<<grid_for((int64_t)S.nslices * 32, 256), 256, 0, s>>>(S.nslices, S.row0, S.nrow, s2n, A.rp,
                                                                            split ? 1 : 0, S.lsh, S.width, w32, lg);
        VEMG_CHECK_LAUNCH();
        VEMG_CHECK_CUDA(cudaMemcpyAsync(&longest, lg.p, sizeof(int), cudaMemcpyDeviceToHost, s));
        total = scan_offsets(w32, S.off, S.nslices, s);   // synchronises
    }
    S.padded = total;
    S.col = ar.alloc<int>(total);
    if (fp32) S.v = ar.alloc<float>(total);
    else S.v = ar.alloc<double>(total);
    void *di = nullptr;
    if (split) {
        if (fp32) di = ar.alloc<float>(n);
        else di = ar.alloc<double>(n);
        *dinv = di;
    }
    if (lsh >= 0) {
        S.rl_wide = longest > 0xffff;
        S.meta = ar.alloc<int4>(S.nslices);
        S.rl = ar.alloc<unsigned>((int64_t)n * (S.rl_wide ? 2 : 1));
    }
    // entries of each group: of earlier colours, and all
    std::vector<unsigned long long> count(2 * (size_t)std::max(ngroups, 1), 0ull);
    if (S.nslices) {
        Scratch<unsigned long long> cnt((int64_t)count.size());
        VEMG_CHECK_CUDA(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long) * count.size(), s));
        const int grid = grid_for((int64_t)S.nslices * 32, 256);
        auto fill = [&](auto *v) {
            using VT = std::remove_pointer_t<decltype(v)>;
            if (lsh >= 0)
                k_sell_deal<VT><<<grid, 256, 0, s>>>(S.nslices, S.lsh, S.row0, S.nrow, S.off, S.width, s2n, n2s, A.rp,
                                                     A.ci, A.v, split, S.col, v, (VT *)di, S.meta, S.rl, S.rl_wide,
                                                     gcol, cnt);
            else
                k_sell_fill<VT><<<grid, 256, 0, s>>>(S.nslices, S.row0, S.nrow, S.off, S.width, s2n, n2s, A.rp, A.ci,
                                                     A.v, S.col, v, cnt);
        };
        if (fp32) fill((float *)S.v);
        else fill((double *)S.v);
        VEMG_CHECK_LAUNCH();
        VEMG_CHECK_CUDA(cudaMemcpyAsync(count.data(), cnt.p, sizeof(unsigned long long) * count.size(),
                                        cudaMemcpyDeviceToHost, s));
        VEMG_CHECK_CUDA(cudaStreamSynchronize(s));
    }
    if (low) {
        low->resize(ngroups);
        all->resize(ngroups);
    }
    for (int g = 0; g < ngroups; ++g) {
        S.nnz += (int64_t)count[2 * g + 1];
        if (low) {
            (*low)[g] = (int64_t)count[2 * g];
            (*all)[g] = (int64_t)count[2 * g + 1];
        }
    }
    return S;
}

__global__ void k_permute_dense(int n, const int *__restrict__ s2n, const double *__restrict__ G, double *Gs) {
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int64_t)n * n) return;
    int a = (int)(t / n), b = (int)(t % n);
    Gs[t] = G[(int64_t)s2n[a] * n + s2n[b]];
}

__global__ void k_to_float(int64_t n, const double *__restrict__ a, float *__restrict__ b) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) b[i] = (float)a[i];
}

// b = a rounded to BF16 (nearest, ties to even); a is overwritten by the same value in FP32
__global__ void k_f2bf(int64_t n, float *__restrict__ a, __nv_bfloat16 *__restrict__ b) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) {
        __nv_bfloat16 h = __float2bfloat16_rn(a[i]);
        b[i] = h;
        a[i] = __bfloat162float(h);
    }
}

// BF16 values of a sliced-ELL matrix, rounded from its FP32 values. The FP32 array keeps the
// rounded values, so that the kernels that read it (the batched solves, the coarse tails, the
// persistent cycle) apply the same operator as the per-phase kernels that read the BF16 array.
static void to_bf16(Arena &ar, Sell &S, cudaStream_t s) {
    __nv_bfloat16 *v = ar.alloc<__nv_bfloat16>(S.padded > 0 ? S.padded : 1);
    if (S.padded > 0) {
        k_f2bf<<<grid_for(S.padded, 256), 256, 0, s>>>(S.padded, (float *)S.v, v);
        VEMG_CHECK_LAUNCH();
    }
    S.vh = v;
}

// bf16: the chain's stored operators get BF16 copies, except on a chain with the near-nullspace
// {1, x, y}, whose coarse operators carry the fourth-order-like part of E~^T A E~ that BF16 values
// lose (measured on the 192x192x48 xy-jittered mesh: 1,593 iterations against 304 with FP32 values);
// it keeps FP32 values
static void layout_chain(Arena &ar, const Chain &C, SChain &S, bool fp32, cudaStream_t s, bool bf16 = false) {
    bf16 = bf16 && C.nsd == 1;
    S.nlev = C.nlev;
    S.direct = C.direct;
    S.singular = C.singular;
    S.fp32 = fp32;
    S.is_bar = C.is_bar;
    std::vector<int *> inv(C.nlev);
    for (int l = 0; l < C.nlev; ++l) {
        const Level &L = C.lv[l];
        inv[l] = ar.alloc<int>(L.A.n);
        k_inverse_perm<<<grid_for(L.A.n, 256), 256, 0, s>>>(L.A.n, L.crow, inv[l]);
        VEMG_CHECK_LAUNCH();
    }
    for (int l = 0; l < C.nlev; ++l) {
        const Level &L = C.lv[l];
        SLevel &T = S.lv[l];
        T.n = L.A.n;
        T.ncolours = L.ncolours;
        T.crow = L.cptr;
        T.A = build_sell(ar, L.A, L.A.n, L.crow, inv[l], L.A.n, L.cptr, fp32, &T.dinv, &T.cslice, s,
                         lanes_shift((double)L.A.n / std::max(L.ncolours, 1), (double)L.A.nnz / std::max(L.A.n, 1) - 1.0, fp32),
                         &T.clow, &T.cnnz);
        if (l + 1 < C.nlev) {
            const Level &N = C.lv[l + 1];
            T.P = build_sell(ar, L.P, L.A.n, L.crow, inv[l + 1], N.A.n, {0, L.A.n}, fp32, nullptr, nullptr, s,
                             lanes_shift(L.A.n, (double)L.P.nnz / std::max(L.A.n, 1), fp32));
            T.PT = build_sell(ar, L.PT, N.A.n, N.crow, inv[l], L.A.n, {0, N.A.n}, fp32, nullptr, nullptr, s,
                              lanes_shift(N.A.n, (double)L.PT.nnz / std::max(N.A.n, 1), fp32));
        }
        if (bf16) {
            to_bf16(ar, T.A, s);
            if (l + 1 < C.nlev) {
                to_bf16(ar, T.P, s);
                to_bf16(ar, T.PT, s);
            }
        }
        size_t es = fp32 ? sizeof(float) : sizeof(double);
        T.x = ar.alloc<char>((int64_t)es * T.n);
        T.b = ar.alloc<char>((int64_t)es * T.n);
        T.r = ar.alloc<char>((int64_t)es * T.n);
    }
    if (C.direct) {
        int n = C.nc;
        S.nc = n;
        S.G = ar.alloc<double>((int64_t)n * n);
        k_permute_dense<<<grid_for((int64_t)n * n, 256), 256, 0, s>>>(n, C.lv[C.nlev - 1].crow, C.G, S.G);
        VEMG_CHECK_LAUNCH();
        if (fp32) {   // FP32 cycles apply the dense inverse in FP32
            S.Gf = ar.alloc<float>((int64_t)n * n);
            k_to_float<<<grid_for((int64_t)n * n, 256), 256, 0, s>>>((int64_t)n * n, S.G, S.Gf);
            VEMG_CHECK_LAUNCH();
        }
    }
}

__global__ void k_outer_order(int n, int mtop, const int *__restrict__ surf_crow, const int *__restrict__ bar_crow,
                              int *s2n) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    s2n[i] = i < mtop ? surf_crow[i] : mtop + bar_crow[i - mtop];
}

__global__ void k_compose(int n, const int *__restrict__ a, const int *__restrict__ b, int off, int *out) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = a[off + b[i]];
}


__global__ void k_iota(int n, int *out) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = i;
}

void build_solve_layout(vemg_hierarchy *h, cudaStream_t s) {
    Arena &ar = h->arena;
    bool fp32 = h->precision != VEMG_PREC_FP64;
    bool bf16 = h->precision == VEMG_PREC_BF16;
    int n = h->n, mt = h->mtop;
    if (!single_chain(h)) {
        layout_chain(ar, h->bar, h->sbar, fp32, s, bf16);
        layout_chain(ar, h->surf, h->ssurf, fp32, s, bf16);
        h->nu = n;
        int *s2n = ar.alloc<int>(n);
        h->s2i = s2n;
        Scratch<int> n2s(n);
        k_outer_order<<<grid_for(n, 256), 256, 0, s>>>(n, mt, h->surf.lv[0].crow, h->bar.lv[0].crow, s2n);
        VEMG_CHECK_LAUNCH();
        k_inverse_perm<<<grid_for(n, 256), 256, 0, s>>>(n, s2n, n2s);
        VEMG_CHECK_LAUNCH();
        Scratch<int> surf_inv(mt);
        k_inverse_perm<<<grid_for(mt, 256), 256, 0, s>>>(mt, h->surf.lv[0].crow, surf_inv);
        VEMG_CHECK_LAUNCH();
        h->Aop = build_sell(ar, h->A, n, s2n, n2s, n, {0, n}, false, nullptr, nullptr, s);
        h->Enon = build_sell(ar, h->E, n - mt, s2n + mt, surf_inv, mt, {0, n - mt}, false, nullptr, nullptr, s);
        h->ETs = build_sell(ar, h->ET, mt, h->surf.lv[0].crow, n2s, n, {0, mt}, false, nullptr, nullptr, s,
                            lanes_shift(mt, (double)h->ET.nnz / std::max(mt, 1), false));
        if (fp32 && h->Enon.padded > 0) {
            // z = E~ y_s + x_bar is formed in FP32 when the V-cycles are FP32 (one conversion per row)
            h->Enon_vf = ar.alloc<float>(h->Enon.padded);
            k_to_float<<<grid_for(h->Enon.padded, 256), 256, 0, s>>>(h->Enon.padded, (const double *)h->Enon.v,
                                                                      h->Enon_vf);
            VEMG_CHECK_LAUNCH();
        }
        h->caller_of = ar.alloc<int>(n);
        k_compose<<<grid_for(n, 256), 256, 0, s>>>(n, h->new2old, s2n, 0, h->caller_of);
        VEMG_CHECK_LAUNCH();
    } else if (h->precond == VEMG_PRECOND_NONE && h->bc == VEMG_NEUMANN) {
        // plain CG: no cycle, the unknowns in their internal order
        h->nu = n;
        int *iota = ar.alloc<int>(n);
        h->s2i = iota;
        k_iota<<<grid_for(n, 256), 256, 0, s>>>(n, iota);
        VEMG_CHECK_LAUNCH();
        h->Aop = build_sell(ar, h->A, n, iota, iota, n, {0, n}, false, nullptr, nullptr, s);
        h->caller_of = ar.alloc<int>(n);
        k_compose<<<grid_for(n, 256), 256, 0, s>>>(n, h->new2old, iota, 0, h->caller_of);
        VEMG_CHECK_LAUNCH();
    } else {
        // one chain whose level 0 is the operator of the unknowns (A_bar for Dirichlet-top, A for
        // the VL_SOR / SA preconditioners); the outer vectors use its level-0 colour order
        const Chain &C = the_chain(h);
        layout_chain(ar, C, h->sbar, fp32, s, bf16);
        int off = h->bc == VEMG_DIRICHLET_TOP ? mt : 0;
        int nb = n - off;
        h->nu = nb;
        const Level &L0 = C.lv[0];
        h->s2i = L0.crow;
        Scratch<int> inv(nb);
        k_inverse_perm<<<grid_for(nb, 256), 256, 0, s>>>(nb, L0.crow, inv);
        VEMG_CHECK_LAUNCH();
        h->Aop = build_sell(ar, L0.A, nb, L0.crow, inv, nb, {0, nb}, false, nullptr, nullptr, s);
        h->caller_of = ar.alloc<int>(nb);
        k_compose<<<grid_for(nb, 256), 256, 0, s>>>(nb, h->new2old + off, L0.crow, 0, h->caller_of);
        VEMG_CHECK_LAUNCH();
    }
    VEMG_CHECK_CUDA(cudaStreamSynchronize(s));
}

}  // namespace vemg
