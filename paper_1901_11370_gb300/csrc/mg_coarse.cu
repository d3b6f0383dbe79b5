// mg_coarse.cu -- dense inverse of a tree's coarsest-level operator on the
// device (Sec. 2.4 of arXiv:1901.11370: the coarsest grid; here it is solved
// exactly).  mg_set_eps needs it for every new coefficient.  Gauss-Jordan
// with pivoting on one host core took 30 ms for the 512 cells of an 8^3
// level, most of a training step that learns eps.
//
// The operator is the 5/7-point row (Sec. 2.2) with homogeneous boundary
// values.  Scaled by the cell volumes it is symmetric and, for eps > 0,
// negative definite -- without a Dirichlet face and lambda only up to the
// constants, which the shift A - sigma 1 V^T (V the volumes, sigma > 0)
// removes.  Row scaling does not change elimination without pivoting, so the
// block Gauss-Jordan inversion below needs none.  Of the bordered matrix
// [A 1; V^T 0] that the host inverts, the solves use the rows of the cells:
// with K = (A - sigma 1 V^T)^-1, v = sum V and A 1 = 0, V^T A = 0 they are
//   K + 1 V^T / (sigma v^2)   and, in the border's column,   1 / v.
// sigma = max |A_ii| / v: the constants move to the operator's own size.  A
// shift of the size of 1 / h^2 alone left K's constant part, or A, with too
// few digits where eps is far from 1 (residual of the solve with 1 .. 10
// times 1e12: 1e-4 of the right-hand side, now 7e-15; bordered 3e-15).
#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "mg_internal.h"
#include "mg_device.cuh"

namespace mg {

constexpr int kPanel = 32;          // pivot block
constexpr int kPanelThreads = 256;
constexpr int kTile = 32;           // update tile, kPanelThreads threads, 2 x 2 values each

// volume of coarsest cell c (block order)
template <int D> __device__ __forceinline__ double coarse_vol(const KParams &P, const TreeCoarse &tc, int c) {
    const BlockDesc &b = P.B[tc.first + c / cells_of<D>(tc.n)];
    const LevelDesc &L = P.L[b.lev];
    if (P.geom != MG_CYL) return L.vol;
    return 2.0 * M_PI * (P.lo[0] + (b.ijk[0] * tc.n + c % tc.n + 0.5) * L.h[0]) * L.h[0] * L.h[1];
}
// sigma from the largest |A_ii| (a single cell that couples to nothing has 0: any shift will do)
__device__ __forceinline__ double coarse_shift(const CoarseInfo *info, double vsum) {
    const double m = __longlong_as_double((long long)info->amax);
    return (m > 0.0 ? m : 1.0) / vsum;
}

// A's row of every coarsest cell, row by row (one thread each; the matrix was
// zeroed): rows and columns in block order, `map` from the cell's global
// index to its row.  flag 2: a coefficient that is not positive (the host
// inverts such a matrix, with pivoting).
template <int D>
__global__ void __launch_bounds__(128) k_coarse_rows(KParams P, TreeCoarse tc, const int *__restrict__ map,
                                                     const double *__restrict__ E, int ld, double *__restrict__ A,
                                                     CoarseInfo *__restrict__ info) {
    pdl_entry();
    const int row = blockIdx.x * blockDim.x + threadIdx.x, C = cells_of<D>(tc.n);
    if (row >= tc.nc) return;
    const BlockDesc &b = P.B[tc.first + row / C];
    const LevelDesc &L = P.L[b.lev];
    int i, j, k;
    cell_of(row % C, tc.n, D, i, j, k);
    const I3 g{b.ijk[0] * tc.n + i, b.ijk[1] * tc.n + j, D == 3 ? b.ijk[2] * tc.n + k : 0};
    const double ri = P.lo[0] + (g.x + 0.5) * L.h[0], ec = E ? E[tc.cell0 + row] : 1.0;
    if (!(ec > 0.0)) info->flag = 2;
    double *a = A + (long long)row * ld;
    double diag = -P.helm;
#pragma unroll
    for (int d = 0; d < D; d++)
#pragma unroll
        for (int s = 0; s < 2; s++) {
            I3 q = g;
            int c = get(g, d) + (s ? 1 : -1);
            bool phys = false;
            if (c < 0 || c >= L.ncell[d]) {
                if (P.bct[2 * d + s] == MG_BC_PERIODIC) c = c < 0 ? c + L.ncell[d] : c - L.ncell[d];
                else phys = true;
            }
            put(q, d, c);
            const int col = phys ? row : map[(q.z * L.ncell[1] + q.y) * L.ncell[0] + q.x];
            double w = 1.0 / (L.h[d] * L.h[d]);
            if (E) {
                const double eo = phys ? ec : E[tc.cell0 + col];
                w *= 2.0 * ec * eo / (ec + eo);
            }
            if (P.geom == MG_CYL && d == 0) w *= (P.lo[0] + (g.x + s) * L.h[0]) / ri;
            if (!phys) {
                if (col == row) continue;  // a periodic extent of one cell: no coupling
                a[col] += w;
                diag -= w;
            } else if (P.bct[2 * d + s] == MG_BC_DIRICHLET) {
                diag -= 2.0 * w;
            }
        }
    a[row] += diag;
    if (tc.singular) atomicMax(&info->amax, (unsigned long long)__double_as_longlong(fabs(diag)));  // >= 0: ordered as integers
}

// The shift of a singular system: - sigma V_c in column c of every row.
template <int D>
__global__ void __launch_bounds__(256) k_coarse_shift(KParams P, TreeCoarse tc, int ld, double vsum,
                                                      const CoarseInfo *__restrict__ info, double *__restrict__ A) {
    pdl_entry();
    const double sigma = coarse_shift(info, vsum);
    const long long total = (long long)tc.nc * tc.nc;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total; e += (long long)gridDim.x * blockDim.x) {
        const int row = (int)(e / tc.nc), c = (int)(e % tc.nc);
        A[(long long)row * ld + c] -= sigma * coarse_vol<D>(P, tc, c);
    }
}

// Step `at` (first row of a pivot block K of nb rows) of the block
// Gauss-Jordan inversion in place, first half: every CTA inverts the pivot
// block for itself (one launch less, and the SMs idle otherwise), then takes
// kTile columns of the pivot rows: R = A_KK^-1 A_K, (A_KK^-1 itself in K's
// columns); and copies its share of the pivot columns.
__global__ void __launch_bounds__(kPanelThreads) k_inv_panel(const double *__restrict__ A, int n, int ld, int at,
                                                             double *__restrict__ R, double *__restrict__ Cc,
                                                             CoarseInfo *__restrict__ info) {
    pdl_entry();
    __shared__ double S[kPanel][kPanel + 1], T[kPanel][kTile + 1];
    const int nb = min(kPanel, n - at), tid = threadIdx.x, c0 = blockIdx.x * kTile;
    for (int e = tid; e < kPanel * kPanel; e += kPanelThreads) {
        const int r = e / kPanel, c = e % kPanel;
        S[r][c] = r < nb && c < nb ? A[(long long)(at + r) * ld + at + c] : (r == c ? 1.0 : 0.0);
        T[r][c] = r < nb && c0 + c < n ? A[(long long)(at + r) * ld + c0 + c] : 0.0;
    }
    for (int e = tid; e < kTile * kPanel; e += kPanelThreads) {  // rows c0 .. of the pivot columns
        const int r = e / kPanel, c = e % kPanel;
        if (c0 + r < n) Cc[(long long)(c0 + r) * kPanel + c] = c < nb ? A[(long long)(c0 + r) * ld + at + c] : 0.0;
    }
    // Gauss-Jordan of S in place: thread (r, cb) holds 4 columns of row r.
    // The warp with the next pivot forms its reciprocal, so that the others'
    // FP64 instructions are one product and four FMAs a step.
    __shared__ double s_ip[2];
    __syncthreads();
    if (tid == 0) s_ip[0] = 1.0 / S[0][0];
    __syncthreads();
    const int r = tid >> 3, cb = (tid & 7) * 4;
    for (int p = 0; p < nb; p++) {
        const double ip = s_ip[p & 1], g = -S[r][p] * ip;
        if (tid == 0 && blockIdx.x == 0 && S[p][p] == 0.0) atomicMax(&info->flag, 1);
        double v[4];
#pragma unroll
        for (int e = 0; e < 4; e++) {
            const int c = cb + e;
            if (r == p) v[e] = c == p ? ip : S[p][c] * ip;
            else v[e] = c == p ? g : fma(g, S[p][c], S[r][c]);
        }
        __syncthreads();
#pragma unroll
        for (int e = 0; e < 4; e++) {
            S[r][cb + e] = v[e];
            if (r == p + 1 && cb + e == p + 1) s_ip[(p + 1) & 1] = 1.0 / v[e];
        }
        __syncthreads();
    }
    double acc[4] = {0, 0, 0, 0};
    for (int p = 0; p < nb; p++)
#pragma unroll
        for (int e = 0; e < 4; e++) acc[e] = fma(S[r][p], T[p][cb + e], acc[e]);
#pragma unroll
    for (int e = 0; e < 4; e++) {
        const int c = c0 + cb + e;
        if (c >= ld) continue;
        const bool own = c >= at && c < at + nb;
        R[(long long)r * ld + c] = own ? S[r][c - at] : (r < nb ? acc[e] : 0.0);
    }
}

// Second half: A_ij - A_iK R_j off the pivot rows and columns, R in the pivot
// rows, - A_iK A_KK^-1 in the pivot columns.  One 32 x 32 tile per CTA: at
// 512 cells that is 256 CTAs of 32K FMAs, which share the SMs' FP64 units
// evenly (64 x 64 tiles left more than half of them idle).
__global__ void __launch_bounds__(kPanelThreads) k_inv_update(double *__restrict__ A, int n, int ld, int at,
                                                              const double *__restrict__ R,
                                                              const double *__restrict__ Cc) {
    pdl_entry();
    __shared__ double X[kTile][kPanel + 1], Y[kPanel][kTile + 1];
    const int nb = min(kPanel, n - at), tid = threadIdx.x, r0 = blockIdx.y * kTile, c0 = blockIdx.x * kTile;
    for (int e = tid; e < kTile * kPanel; e += kPanelThreads) {
        const int a = e / kPanel, b = e % kPanel;
        X[a][b] = r0 + a < n ? Cc[(long long)(r0 + a) * kPanel + b] : 0.0;
        Y[a][b] = c0 + b < ld ? R[(long long)a * ld + c0 + b] : 0.0;
    }
    __syncthreads();
    const int tr = tid >> 4, tc = tid & 15;  // values (tr + 16 i, tc + 16 j)
    double s[2][2] = {{0, 0}, {0, 0}};
    for (int p = 0; p < nb; p++) {
        const double x0 = X[tr][p], x1 = X[tr + 16][p], y0 = Y[p][tc], y1 = Y[p][tc + 16];
        s[0][0] = fma(x0, y0, s[0][0]);
        s[0][1] = fma(x0, y1, s[0][1]);
        s[1][0] = fma(x1, y0, s[1][0]);
        s[1][1] = fma(x1, y1, s[1][1]);
    }
#pragma unroll
    for (int i = 0; i < 2; i++)
#pragma unroll
        for (int j = 0; j < 2; j++) {
            const int row = r0 + tr + 16 * i, col = c0 + tc + 16 * j;
            if (row >= n || col >= n) continue;
            double *a = A + (long long)row * ld + col;
            const bool prow = row >= at && row < at + nb, pcol = col >= at && col < at + nb;
            if (prow) *a = R[(long long)(row - at) * ld + col];
            else *a = pcol ? -s[i][j] : *a - s[i][j];
        }
}

// The inverse (rows of nc, stride ld) into the rows of ns values that the
// coarsest solves read; singular: plus 1 V^T / (sigma v^2), 1 / v in the
// border's column.
template <int D>
__global__ void __launch_bounds__(256) k_inv_store(KParams P, TreeCoarse tc, const double *__restrict__ A, int ld,
                                                   double vsum, const CoarseInfo *__restrict__ info,
                                                   double *__restrict__ minv) {
    pdl_entry();
    const long long total = (long long)tc.nc * tc.ns;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total; e += (long long)gridDim.x * blockDim.x) {
        const int row = (int)(e / tc.ns), c = (int)(e % tc.ns);
        if (c == tc.nc) {
            minv[e] = 1.0 / vsum;
            continue;
        }
        double v = A[(long long)row * ld + c];
        if (tc.singular) v += coarse_vol<D>(P, tc, c) / vsum / (coarse_shift(info, vsum) * vsum);
        minv[e] = v;
    }
}

static bool calloc_dev(void **p, size_t bytes) {
    if (*p) return true;
    if (cudaMalloc(p, bytes) == cudaSuccess) return true;
    cudaGetLastError();
    *p = nullptr;
    return false;
}

template <int D> static int inverse_d(mg_tree *t) {
    const TreeCoarse &tc = t->tcoarse[0];
    const LevelHost &L = t->lev[0];
    const int nc = tc.nc, ld = (nc + kTile - 1) / kTile * kTile;
    if (!t->d_cwork) {
        std::vector<int> map((size_t)L.ncell[0] * L.ncell[1] * L.ncell[2]);
        const int C = cells_of<D>(L.n), n = L.n;
        for (int b = 0; b < tc.nb; b++)
            for (int c = 0; c < C; c++) {
                const BlockDesc &B = t->blocks[tc.first + b];
                const int x = B.ijk[0] * n + c % n, y = B.ijk[1] * n + c / n % n, z = D == 3 ? B.ijk[2] * n + c / (n * n) : 0;
                map[((size_t)z * L.ncell[1] + y) * L.ncell[0] + x] = b * C + c;
            }
        if (!calloc_dev((void **)&t->d_crow, sizeof(int) * map.size()) || !calloc_dev((void **)&t->d_cinfo, sizeof(CoarseInfo)) ||
            !calloc_dev((void **)&t->d_minv, sizeof(double) * (size_t)t->minv_total) ||
            !calloc_dev((void **)&t->d_cwork, sizeof(double) * ((size_t)nc * ld + 2 * (size_t)kPanel * ld)))
            return 1;
        if (upload(t->d_crow, map.data(), sizeof(int) * map.size(), t->stream) != cudaSuccess)
            return check_cuda("coarsest inverse");
    }
    double vsum = 0;
    if (tc.singular) {
        for (int x = 0; x < L.ncell[0]; x++) {
            double V = 1.0;
            for (int d = 0; d < D; d++) V *= L.h[d];
            if (t->geom == MG_CYL) V = 2.0 * M_PI * (t->lo[0] + (x + 0.5) * L.h[0]) * L.h[0] * L.h[1];
            vsum += V * L.ncell[1] * L.ncell[2];
        }
    }
    const KParams P = kparams(t, 1);
    double *A = t->d_cwork, *R = A + (size_t)nc * ld, *Cc = R + (size_t)kPanel * ld;
    cudaMemsetAsync(A, 0, sizeof(double) * (size_t)nc * ld, t->stream);
    cudaMemsetAsync(t->d_cinfo, 0, sizeof(CoarseInfo), t->stream);
    ++t->launches;
    launch_k(k_coarse_rows<D>, (nc + 127) / 128, 128, 0, t->stream, P, tc, (const int *)t->d_crow,
             t->var_eps ? (const double *)t->f64.E : (const double *)nullptr, ld, A, t->d_cinfo);
    const int elems = (int)std::max<long long>(1, std::min<long long>(((long long)nc * tc.ns + 255) / 256, 8LL * t->nsm));
    if (tc.singular) {
        ++t->launches;
        launch_k(k_coarse_shift<D>, elems, 256, 0, t->stream, P, tc, ld, vsum, (const CoarseInfo *)t->d_cinfo, A);
    }
    const int tiles = ld / kTile;
    for (int at = 0; at < nc; at += kPanel) {
        t->launches += 2;
        launch_k(k_inv_panel, tiles, kPanelThreads, 0, t->stream, (const double *)A, nc, ld, at, R, Cc, t->d_cinfo);
        launch_k(k_inv_update, dim3(tiles, tiles), kPanelThreads, 0, t->stream, A, nc, ld, at, (const double *)R,
                 (const double *)Cc);
    }
    ++t->launches;
    launch_k(k_inv_store<D>, elems, 256, 0, t->stream, P, tc, (const double *)A, ld, vsum,
             (const CoarseInfo *)t->d_cinfo, t->d_minv);
    int flag = 0;
    if (cudaMemcpyAsync(&flag, &t->d_cinfo->flag, sizeof(int), cudaMemcpyDeviceToHost, t->stream) != cudaSuccess ||
        cudaStreamSynchronize(t->stream) != cudaSuccess)
        return check_cuda("coarsest inverse");
    const int rc = check_cuda("coarsest inverse");
    return rc ? rc : (flag ? 1 : 0);  // zero pivot or eps <= 0: the host's pivoting inversion decides
}

void coarse_inverse_free(mg_tree *t) {
    cudaFree(t->d_cwork);
    cudaFree(t->d_crow);
    cudaFree(t->d_cinfo);
    t->d_cwork = nullptr;
    t->d_crow = nullptr;
    t->d_cinfo = nullptr;
}

// The scratch (as large as the inverse) stays while eps may be set again; a
// constant coefficient is inverted once, when the tree is made.  Up to 80
// cells the host's elimination is sooner done than the launches: set_eps with
// 60 cells 112 against 155 us, 64 cells 120 / 161, 100 cells 296 / 235.
int coarse_inverse_device(mg_tree *t) {
    if (t->is_batch || t->tcoarse.size() != 1 || t->tcoarse[0].bt_n || t->tcoarse[0].nc <= 80) return 1;
    const int rc = t->dim == 2 ? inverse_d<2>(t) : inverse_d<3>(t);
    if (!t->var_eps || rc > 0) coarse_inverse_free(t);
    return rc;
}

}  // namespace mg
