// mg_bottom.cu -- the lower levels of a V-cycle or FMG (Teunissen & Keppens,
// arXiv:1901.11370, Sec. 2.4) in one launch of one thread-block cluster.
//
// Every level up to the base grid covers the whole domain, so the levels
// 0 .. top of a tree (top at most the base grid) are complete uniform grids.
// The launch-by-launch cycle spends 3 to 6 us on each of their colour
// sweeps, transfers and ghost fills whatever the level's size (launch and
// dependent-load latency).  Here a cluster of up to 16 CTAs keeps x, f and
// the FAS copy of all these levels in shared memory, as dense padded slabs,
// and runs the whole leg: smoothing, restriction, FAS right-hand sides, the
// exact coarsest solve, prolongation.  A CTA owns a slab of every level
// (slabs of level l are those of level 0 times 2^l, so children and parents
// share a CTA); the cells beside a slab face are pushed into the neighbour's
// halo with st.shared::cluster when they change, and one cluster barrier
// follows each colour.  The ghost rules of Sec. 2.6 are applied by the
// thread that updates the cell beside the boundary, after every colour as in
// the sweep kernels, so the cycle is the same up to rounding order.
//
// What bounds it: the latency of a step, about 1.0 us for a half-sweep of a
// level of up to 16^3 cells in FP32 (arithmetic 0.2, block barrier and face
// stores 0.4, cluster barrier with the remote stores' release 0.3; the
// barrier alone takes 480 cycles with release and acquire, 130 without) and
// 1.3 us at 32^3; in FP64 the SM's FP64 unit adds to it (5 us at 32^3,
// 1.0 us at 64^2).  One launch replaces the 8 sweeps, 3 transfers and ghost
// fills of each level at 3.5 to 6 us apiece: the 64^2 FP64 solve went from
// 1448 to 828 us (406 launches to 40), the 1152 x 864 Helmholtz step from
// 2737 to 1666 us, the 160 x 96 x 48 solve from 3065 to 1871 us, the
// cleaning step with its adjoint on 64^3 from 12.5 to 7.4 ms.  Clusters of
// 8 instead of 16 CTAs: 1867 and 1942 us for the second and third.
#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "mg_internal.h"
#include "mg_device.cuh"

namespace mg {

constexpr int kBotThreads = 512;
constexpr int kBotPer = 8;                 // colour cells a thread may own on a level
constexpr int kBotMap = 1024;              // blocks of the top level whose map is kept in shared memory
constexpr size_t kBotSmem = 220 * 1024;    // dynamic shared memory of one CTA (static part beside it)

// x / d for x d < 2^32, with m = ceil(2^32 / d)
__device__ __forceinline__ unsigned bot_magic(int d) { return d == 1 ? 0u : 0xffffffffu / (unsigned)d + 1u; }
__device__ __forceinline__ int bot_div(int x, unsigned m) { return m ? (int)__umulhi((unsigned)x, m) : x; }

__device__ __forceinline__ void cluster_sync() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// cluster address of the place that p has in this CTA, in CTA `rank`
__device__ __forceinline__ unsigned rank_addr(const void *p, int rank) {
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_cluster(unsigned a, float v) { asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory"); }
__device__ __forceinline__ void st_cluster(unsigned a, double v) { asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory"); }

// Division magics of one level, computed once per launch: a, a / 2, a / 4, b, b / 2
// and a / 32 cells.
struct BotMagic {
    unsigned a, ha, qa, b, hb, hr;
};

// One CTA's slab of one level.  Local dimensions: a (whole in every CTA), b
// and p (cut over the cluster); in 2D b has one cell and no neighbours.
template <class T, int D> struct BotLev {
    int l, A, Bn, Pn, gb, gp;  // cells of the slab, its first global b and p
    int SA, SP;                // strides of the padded array
    int tb, tp;                // cells of the lower neighbour's slab (its upper halo starts there)
    T *X, *F, *V;
    const T *W;                // coefficients: [slot][p][b][a] of the whole level, 2D faces then 1 / diagonal
    long long wn;              // cells of the whole level (slot stride)
    int NB;                    // whole level's b cells
    __device__ __forceinline__ int at(int a, int b, int p) const { return (p + 1) * SP + (D == 3 ? (b + 1) * SA : 0) + a + 1; }
    // f has the strides of x without the halo planes of p, so that one index serves both: fat = at - SP
    __device__ __forceinline__ int fat(int a, int b, int p) const { return at(a, b, p) - SP; }
    __device__ __forceinline__ long long wat(int a, int b, int p) const {
        return ((long long)(gp + p) * NB + gb + b) * A + a;
    }
};

template <class T, int D, bool VAR> struct Bottom {
    const KParams &P;
    const BotPlan &B;
    const Fields<T> &G;
    const T *Wd;
    const LevelDesc *L;  // levels 0 .. top, in shared memory
    const BotMagic *M;
    T *base;
    double *part;  // the ranks' partial sums (singular problems)
    double *r;     // coarsest residual and the steps of its solve
    const double *fd_tab, *fd_g;  // eigenvectors along a and b (shared memory); solves along p (global)
    int tid, nth, rank;
    int b0, bl, p0, pl, tb, tp;      // this CTA's slab of level 0 and the lower neighbours' sizes
    int rbl, rbh, rpl, rph;          // ranks beside the slab faces, -1: physical boundary
    bool pera;
    T omega;
    const int *bmap;  // block map of the top level (a copy in shared memory where it fits)

    __device__ __forceinline__ BotLev<T, D> lev(int l) const {
        BotLev<T, D> q;
        q.l = l;
        q.A = B.n0[0] << l;
        q.Bn = D == 3 ? bl << l : 1;
        q.Pn = pl << l;
        q.gb = D == 3 ? b0 << l : 0;
        q.gp = p0 << l;
        q.SA = q.A + 2;
        q.SP = q.SA * (D == 3 ? (B.mb << l) + 2 : 1);
        q.tb = tb << l;
        q.tp = tp << l;
        q.X = base + B.offx[l];
        q.F = base + B.offf[l];
        q.V = base + B.offv[l];
        q.NB = D == 3 ? B.n0[1] << l : 1;
        q.wn = (long long)q.A * q.NB * (B.n0[2] << l);
        q.W = VAR ? Wd + B.woff[l] : nullptr;
        return q;
    }
    // value of the physical ghost beside a cell (Sec. 2.6); i: local dimension, s: side
    __device__ __forceinline__ T ghost(const BotLev<T, D> &q, int i, int s, T v, int ga, int gb, int gp) const {
        const int d = i == 0 ? B.perm[0] : i == 1 ? B.perm[1] : B.perm[2], face = 2 * d + s;
        double a = 0.0;
        if (!P.homog) {
            const LevelDesc &M = L[q.l];
            if (M.bc_off[face] < 0) {
                a = P.bcv[face];
            } else {
                const int x = B.perm[0] == 0 ? ga : (B.perm[1] == 0 ? gb : gp);
                const int y = B.perm[0] == 1 ? ga : (B.perm[1] == 1 ? gb : gp);
                const int z = D == 2 ? 0 : (B.perm[0] == 2 ? ga : (B.perm[1] == 2 ? gb : gp));
                const int t1 = d == 0 ? y : x, t2 = D == 2 ? 0 : (d == 2 ? y : z);
                a = P.bcplanes[M.bc_off[face] + t1 + (long long)M.ncell[d == 0 ? 1 : 0] * t2];
            }
        }
        return phys_ghost<T>(P, L[q.l], face, v, a);
    }
    // After cells of array Y changed (colour 0 / 1, or -1 for all), every
    // ghost and halo value they feed is stored: one item per cell beside a
    // slab face.  The faces take whole
    // warps, so that no warp meets two of them.  Kept out of the cell loops:
    // there some lane of nearly every warp sits beside a face, and every
    // warp paid for the ghost code.
    struct Item {
        int src;       // padded index of the cell, -1: none
        unsigned dst;  // where the value goes: padded index, or address in another CTA
        T s, g;
        int kind;      // 0: copy within the slab, 1: s x + g within the slab, 2: copy to another CTA
    };
    __device__ __forceinline__ int nfaces(const BotLev<T, D> &q, bool half) const {
        const int ca = half ? q.A >> 1 : q.A, cb = D == 3 && half ? q.Bn >> 1 : q.Bn, cp = D == 2 && half ? q.Pn >> 1 : q.Pn;
        return 2 * (((cb * cp + 31) & ~31) + (D == 3 ? (ca * q.Pn + 31) & ~31 : 0) + ((ca * q.Bn + 31) & ~31));
    }
    __device__ __forceinline__ Item item(const BotLev<T, D> &q, T *Y, int colour, int t) const {
        const bool hf = colour >= 0;  // half the cells of a face
        const int ca = hf ? q.A >> 1 : q.A, cb = D == 3 && hf ? q.Bn >> 1 : q.Bn;
        const int cp = D == 2 && hf ? q.Pn >> 1 : q.Pn;
        const int na = cb * cp, nb = D == 3 ? ca * q.Pn : 0, np = ca * q.Bn;  // items of one a, b, p face
        const int ra = (na + 31) & ~31, rb = (nb + 31) & ~31, rp = (np + 31) & ~31;
        const int par = (colour + q.gb + q.gp) & 1;
        const unsigned mA = hf ? M[q.l].ha : M[q.l].a;
        int a, b = 0, p, i, sd, rank, dim, dst;
        if (t < 2 * ra) {
            sd = t >= ra;
            const int u = t - sd * ra;
            if (u >= na) return Item{-1, 0u, (T)1, (T)0, 0};
            dim = 0;
            a = sd ? q.A - 1 : 0;
            if (D == 3) {
                p = bot_div(u, hf ? M[q.l].hb : M[q.l].b);
                b = u - p * cb;
                if (hf) b = 2 * b + ((par + p + a) & 1);
            } else {
                p = hf ? 2 * u + ((par + a) & 1) : u;
            }
            i = q.at(a, b, p);
            rank = pera ? -2 : -1;
            dst = pera ? (sd ? i - q.A : i + q.A) : (sd ? i + 1 : i - 1);
        } else if (D == 3 && t < 2 * (ra + rb)) {
            const int w = t - 2 * ra;
            sd = w >= rb;
            const int u = w - sd * rb;
            if (u >= nb) return Item{-1, 0u, (T)1, (T)0, 0};
            dim = 1;
            p = bot_div(u, mA);
            b = sd ? q.Bn - 1 : 0;
            a = u - p * ca;
            if (hf) a = 2 * a + ((par + b + p) & 1);
            i = q.at(a, b, p);
            rank = sd ? rbh : rbl;
            dst = rank < 0 ? (sd ? i + q.SA : i - q.SA) : q.at(a, sd ? -1 : q.tb, p);
        } else {
            const int w = t - 2 * (ra + rb);
            sd = w >= rp;
            const int u = w - sd * rp;
            if (u >= np) return Item{-1, 0u, (T)1, (T)0, 0};
            dim = 2;
            b = bot_div(u, mA);
            p = sd ? q.Pn - 1 : 0;
            a = u - b * ca;
            if (hf) a = 2 * a + ((par + b + p) & 1);
            i = q.at(a, b, p);
            rank = sd ? rph : rpl;
            dst = rank < 0 ? (sd ? i + q.SP : i - q.SP) : q.at(a, b, sd ? -1 : q.tp);
        }
        if (rank >= 0) return Item{i, rank_addr(Y + dst, rank), (T)1, (T)0, 2};
        Item it{i, (unsigned)dst, (T)1, (T)0, 0};
        if (rank == -1) {  // physical face (Sec. 2.6): Dirichlet 2a - x, Neumann x -/+ h b, axis x
            const int d = dim == 0 ? B.perm[0] : (dim == 1 ? B.perm[1] : B.perm[2]);
            it.s = P.bct[2 * d + sd] == MG_BC_DIRICHLET ? (T)-1 : (T)1;
            if (!P.homog) it.g = ghost(q, dim, sd, (T)0, a, q.gb + b, q.gp + p);
            it.kind = it.s == (T)1 && it.g == (T)0 ? 0 : 1;
        }
        return it;
    }
    __device__ __forceinline__ void send(const Item &it, T *Y) const {
        if (it.src < 0) return;
        const T v = Y[it.src];
        if (it.kind == 2) st_cluster(it.dst, v);
        else Y[it.dst] = it.kind ? it.s * v + it.g : v;
    }
    // the same face by face, without the items' indices kept
    __device__ __forceinline__ void faces(const BotLev<T, D> &q, T *Y, int colour) const {
        const bool hf = colour >= 0;
        const int par = (colour + q.gb + q.gp) & 1;
        const int ca = hf ? q.A >> 1 : q.A;
        const unsigned mA = hf ? M[q.l].ha : M[q.l].a;
        {  // a faces: both ends of a row
            const int cb = D == 3 && hf ? q.Bn >> 1 : q.Bn, cp = D == 2 && hf ? q.Pn >> 1 : q.Pn, n = cb * cp;
            const unsigned mC = hf ? M[q.l].hb : M[q.l].b;
            for (int u = tid; u < 2 * n; u += nth) {
                const int sd = u >= n, w = u - sd * n, a = sd ? q.A - 1 : 0;
                int b = 0, p;
                if (D == 3) {
                    p = bot_div(w, mC);
                    b = w - p * cb;
                    if (hf) b = 2 * b + ((par + p + a) & 1);
                } else {
                    p = hf ? 2 * w + ((par + a) & 1) : w;
                }
                const int i = q.at(a, b, p);
                const T v = Y[i];
                if (pera) Y[sd ? i - q.A : i + q.A] = v;
                else Y[sd ? i + 1 : i - 1] = ghost(q, 0, sd, v, a, q.gb + b, q.gp + p);
            }
        }
#pragma unroll
        for (int sd = 0; sd < 2; sd++) {
            if (D == 3) {
                const int n = ca * q.Pn, b = sd ? q.Bn - 1 : 0, rk = sd ? rbh : rbl, st = sd ? q.SA : -q.SA;
                const unsigned far = rk < 0 ? 0u : rank_addr(Y + q.at(0, sd ? -1 : q.tb, 0), rk);
                for (int u = tid; u < n; u += nth) {
                    const int p = bot_div(u, mA);
                    int a = u - p * ca;
                    if (hf) a = 2 * a + ((par + b + p) & 1);
                    const int i = q.at(a, b, p);
                    const T v = Y[i];
                    if (rk < 0) Y[i + st] = ghost(q, 1, sd, v, a, q.gb + b, q.gp + p);
                    else st_cluster(far + (unsigned)(sizeof(T) * (p * q.SP + a)), v);
                }
            }
            {
                const int n = ca * q.Bn, p = sd ? q.Pn - 1 : 0, rk = sd ? rph : rpl, st = sd ? q.SP : -q.SP;
                const unsigned far = rk < 0 ? 0u : rank_addr(Y + q.at(0, 0, sd ? -1 : q.tp), rk);
                for (int u = tid; u < n; u += nth) {
                    const int b = bot_div(u, mA);
                    int a = u - b * ca;
                    if (hf) a = 2 * a + ((par + b + p) & 1);
                    const int i = q.at(a, b, p);
                    const T v = Y[i];
                    if (rk < 0) Y[i + st] = ghost(q, 2, sd, v, a, q.gb + b, q.gp + p);
                    else st_cluster(far + (unsigned)(sizeof(T) * (b * q.SA + a)), v);
                }
            }
        }
    }
    // the cells' own stores are done, then what they feed, then the cluster's barrier
    __device__ __forceinline__ void publish(const BotLev<T, D> &q, T *Y, int colour) const {
        __syncthreads();
        faces(q, Y, colour);
        cluster_sync();
    }
    __device__ __forceinline__ T ih(int l, int i) const { return lv_ih<T>(L[l], B.perm[i]); }
    // L x - lambda x at a cell of level q, in differences: their rounding
    // follows w |dx|, that of a sum form w |x|
    __device__ __forceinline__ T lap(const BotLev<T, D> &q, int a, int b, int p, T w0, T w1, T w2) const {
        const T *x = q.X + q.at(a, b, p);
        const T xc = x[0];
        if (VAR) {
            const T *w = q.W + q.wat(a, b, p);
            T s = w[0] * (x[-1] - xc);
            s += w[q.wn] * (x[1] - xc);
            if (D == 3) {
                s += w[2 * q.wn] * (x[-q.SA] - xc);
                s += w[3 * q.wn] * (x[q.SA] - xc);
            }
            s += w[(2 * D - 2) * q.wn] * (x[-q.SP] - xc);
            s += w[(2 * D - 1) * q.wn] * (x[q.SP] - xc);
            return s - kp_helm<T>(P) * xc;
        }
        T s = w0 * (x[-1] - xc);
        s += w0 * (x[1] - xc);
        if (D == 3) {
            s += w1 * (x[-q.SA] - xc);
            s += w1 * (x[q.SA] - xc);
        }
        s += w2 * (x[-q.SP] - xc);
        s += w2 * (x[q.SP] - xc);
        return s - kp_helm<T>(P) * xc;
    }
    // the local Gauss-Seidel solution at padded index i (Sec. 2.2); wi: its coefficient index
    __device__ __forceinline__ T local_at(const BotLev<T, D> &q, int i, int wi, T w0, T w1, T w2, T idiag) const {
        const T *x = q.X + i;
        const T f = q.F[i - q.SP];
        if (VAR) {
            const T *w = q.W + wi;
            T num = w[0] * x[-1];
            num += w[q.wn] * x[1];
            if (D == 3) {
                num += w[2 * q.wn] * x[-q.SA];
                num += w[3 * q.wn] * x[q.SA];
            }
            num += w[(2 * D - 2) * q.wn] * x[-q.SP];
            num += w[(2 * D - 1) * q.wn] * x[q.SP];
            return (num - f) * w[2 * D * q.wn];
        }
        T num = w0 * (x[-1] + x[1]);
        if (D == 3) num += w1 * (x[-q.SA] + x[q.SA]);
        num += w2 * (x[-q.SP] + x[q.SP]);
        return (num - f) * idiag;
    }
    // Red-black sweeps of level q where a thread owns at most PER colour
    // cells: it keeps the padded index of its cell pairs (and of at most two
    // face items per colour) through the whole phase, so that a half-sweep is
    // loads, arithmetic, stores and the barrier -- the index arithmetic took
    // half of a small level's time.  Cells of the other colour are not
    // written, so the loads of several cells go before their stores.
    template <int PER> __device__ void smooth_gs(const BotLev<T, D> &q, int steps, T w0, T w1, T w2, T idiag) const {
        const int HA = q.A >> 1, ncol = HA * q.Bn * q.Pn, par = q.gb + q.gp;
        const BotMagic mg = M[q.l];
        int pair[PER];  // 2 at(2m, b, p) + parity of b + p (a thread without a cell repeats its last one)
        // this thread's cells, and those of its warp's first lane: a warp past
        // its last cell skips the arithmetic (FP64 instructions would occupy
        // the SM's unit whatever becomes of them)
        const int own = (ncol - tid + nth - 1) / nth, wown = (ncol - (tid & ~31) + nth - 1) / nth;
        int wi[VAR ? PER : 1];
#pragma unroll
        for (int e = 0; e < PER; e++) {
            const int c = min(tid + e * nth, ncol - 1);
            int row, m;
            if (HA >= 32 && !(HA & 15)) {
                // a warp takes 16 pairs of each of two rows (their count is
                // even above level 0): the rows have opposite parity, so
                // their cells fall into different banks
                const int rest = c >> 5, hb = HA >> 4, rp = bot_div(rest, mg.hr);
                m = (rest - rp * hb) * 16 + (c & 15);
                row = 2 * rp + ((c >> 4) & 1);
            } else {
                row = bot_div(c, mg.ha);
                m = c - row * HA;
            }
            const int p = bot_div(row, mg.b), b = row - p * q.Bn;
            pair[e] = 2 * q.at(2 * m, b, p) + ((b + p + par) & 1);
            if (VAR) wi[e] = (int)q.wat(2 * m, b, p);
        }
        constexpr int kItems = PER <= 4 ? 2 : 0;  // face items a thread keeps per colour (registers allow none above)
        const int nf = nfaces(q, true);
        const bool kept = nf <= kItems * nth;
        Item it[2][kItems ? kItems : 1];
#pragma unroll
        for (int k = 0; k < kItems; k++) {
            it[0][k] = it[1][k] = Item{-1, 0u, (T)1, (T)0, 0};
            if (kept && tid + k * nth < nf) {
                it[0][k] = item(q, q.X, 0, tid + k * nth);
                it[1][k] = item(q, q.X, 1, tid + k * nth);
            }
        }
        constexpr int kBatch = PER < 4 ? PER : (sizeof(T) == 4 ? 4 : 2);
        for (int st = 0; st < steps; st++)
#pragma unroll
            for (int s = 0; s < 2; s++) {
#pragma unroll
                for (int e0 = 0; e0 < PER; e0 += kBatch) {
                    if (e0 >= wown) break;
                    T v[kBatch];
#pragma unroll
                    for (int e = 0; e < kBatch; e++) {
                        const int k = pair[e0 + e], o = (s + k) & 1;
                        v[e] = local_at(q, (k >> 1) + o, VAR ? wi[VAR ? e0 + e : 0] + o : 0, w0, w1, w2, idiag);
                    }
#pragma unroll
                    for (int e = 0; e < kBatch; e++) {
                        const int k = pair[e0 + e];
                        if (e0 + e < own) q.X[(k >> 1) + ((s + k) & 1)] = v[e];
                    }
                }
                __syncthreads();
                if (kept) {
#pragma unroll
                    for (int k = 0; k < kItems; k++) send(it[s][k], q.X);
                } else {
                    faces(q, q.X, s);
                }
                cluster_sync();
            }
    }
    __device__ void smooth(int l, int steps) const {
        const BotLev<T, D> q = lev(l);
        const T w0 = ih(l, 0), w1 = ih(l, 1), w2 = ih(l, 2), idiag = lv_idiag<T>(L[l]);
        if (B.jac) {
            T *J = base + B.offj;
            const int cells = q.A * q.Bn * q.Pn, all = q.SP * (q.Pn + 2);
            for (int s = 0; s < steps; s++) {
                for (int c = tid; c < cells; c += nth) {
                    const int row = bot_div(c, M[l].a), a = c - row * q.A, p = bot_div(row, M[l].b), b = row - p * q.Bn;
                    const int i = q.at(a, b, p);
                    const T xc = q.X[i];
                    J[i] = xc + omega * (local_at(q, i, VAR ? (int)q.wat(a, b, p) : 0, w0, w1, w2, idiag) - xc);
                }
                publish(q, J, -1);
                for (int i = tid; i < all; i += nth) q.X[i] = J[i];
                cluster_sync();
            }
            return;
        }
        const int per = ((q.A >> 1) * q.Bn * q.Pn + nth - 1) / nth;
        if (per <= 1) smooth_gs<1>(q, steps, w0, w1, w2, idiag);
        else if (per <= 2) smooth_gs<2>(q, steps, w0, w1, w2, idiag);
        else if (per <= 4) smooth_gs<4>(q, steps, w0, w1, w2, idiag);
        else smooth_gs<kBotPer>(q, steps, w0, w1, w2, idiag);
    }
    // from level l to l - 1 (Sec. 2.3, 2.4): means of x and of the residual,
    // then f^H += L x^H and v_old = x^H (ghosts and halos included)
    __device__ void restrict_to(int l) const {
        const BotLev<T, D> q = lev(l), h = lev(l - 1);
        const T w0 = ih(l, 0), w1 = ih(l, 1), w2 = ih(l, 2), helm = kp_helm<T>(P);
        const unsigned mA = M[l - 1].a, mB = M[l - 1].b;
        const int cells = h.A * h.Bn * h.Pn;
        for (int c = tid; c < cells; c += nth) {
            const int row = bot_div(c, mA), a = c - row * h.A, p = bot_div(row, mB), b = row - p * h.Bn;
            const int fa = 2 * a, fb = D == 3 ? 2 * b : 0, fp = 2 * p;
            T sx = 0, sr = 0;
            if (sizeof(T) == 8 && !VAR) {
                // FP64: the Laplacians of the 2^D children share their inner
                // faces, whose fluxes cancel: sum_d w_d sum (outer neighbour
                // in d - child), the differences kept (see k_restrict_tma).
                // 8 instead of 16 FP64 instructions a child.
                T oa = 0, ob = 0, op = 0;
                const T *x = q.X + q.at(fa, fb, fp);
                const T *f = q.F + q.fat(fa, fb, fp);
#pragma unroll
                for (int e = 0; e < (D == 3 ? 2 : 1); e++)
#pragma unroll
                    for (int g = 0; g < 2; g++) {  // the row of children at b + e, p + g
                        const T *y = x + e * q.SA + g * q.SP;
                        const T y0 = y[0], y1 = y[1];
                        sx += y0 + y1;
                        oa += (y[-1] - y0) + (y[2] - y1);
                        if (D == 3) {
                            const T *o = y + (e ? q.SA : -q.SA);
                            ob += (o[0] - y0) + (o[1] - y1);
                        }
                        const T *o = y + (g ? q.SP : -q.SP);
                        op += (o[0] - y0) + (o[1] - y1);
                        const T *fr = f + e * q.SA + g * q.SP;
                        sr += fr[0] + fr[1];
                    }
                T s = fma(helm, sx, sr);
                s = fma(-w0, oa, s);
                if (D == 3) s = fma(-w1, ob, s);
                sr = fma(-w2, op, s);
            } else {
#pragma unroll
                for (int ch = 0; ch < (1 << D); ch++) {
                    const int ca = fa + (ch & 1), cb = D == 3 ? fb + ((ch >> 1) & 1) : 0, cp = fp + (ch >> (D - 1));
                    sx += q.X[q.at(ca, cb, cp)];
                    sr += q.F[q.fat(ca, cb, cp)] - lap(q, ca, cb, cp, w0, w1, w2);
                }
            }
            h.X[h.at(a, b, p)] = sx * (T)(1.0 / (1 << D));
            h.F[h.fat(a, b, p)] = sr * (T)(1.0 / (1 << D));
        }
        publish(h, h.X, -1);
        fas(h, l - 1);
        const int all = h.SP * (h.Pn + 2);
        for (int i = tid; i < all; i += nth) h.V[i] = h.X[i];
        cluster_sync();
    }
    __device__ __forceinline__ void fas(const BotLev<T, D> &h, int l) const {
        const T w0 = ih(l, 0), w1 = ih(l, 1), w2 = ih(l, 2);
        const unsigned mA = M[l].a, mB = M[l].b;
        const int cells = h.A * h.Bn * h.Pn;
        for (int c = tid; c < cells; c += nth) {
            const int row = bot_div(c, mA), a = c - row * h.A, p = bot_div(row, mB), b = row - p * h.Bn;
            h.F[h.fat(a, b, p)] += lap(h, a, b, p, w0, w1, w2);
        }
    }
    // x_l += P(x_{l-1} - v_old) (Sec. 2.3)
    __device__ void prolong_to(int l) const {
        const BotLev<T, D> q = lev(l), h = lev(l - 1);
        const int all = h.SP * (h.Pn + 2);
        for (int i = tid; i < all; i += nth) h.V[i] = h.X[i] - h.V[i];
        __syncthreads();
        const unsigned mA = M[l].a, mB = M[l].b;
        const int cells = q.A * q.Bn * q.Pn;
        for (int c = tid; c < cells; c += nth) {
            const int row = bot_div(c, mA), a = c - row * q.A, p = bot_div(row, mB), b = row - p * q.Bn;
            const T *v = h.V + h.at(a >> 1, D == 3 ? b >> 1 : 0, p >> 1);  // slabs start at even cells: local parity is global
            T nbs = v[(a & 1) ? 1 : -1];
            if (D == 3) nbs += v[(b & 1) ? h.SA : -h.SA];
            nbs += v[(p & 1) ? h.SP : -h.SP];
            const T val = D == 2 ? ((T)2 * v[0] + nbs) * (T)0.25 : (v[0] + nbs) * (T)0.25;
            q.X[q.at(a, b, p)] += val;
        }
        publish(q, q.X, -1);
    }
    // row of a coarsest cell in the inverse (block order)
    __device__ __forceinline__ int coarse_row(int a, int b, int p) const {
        const int g0 = a, g1 = b, g2 = p;
        const int x = B.perm[0] == 0 ? g0 : (B.perm[1] == 0 ? g1 : g2);
        const int y = B.perm[0] == 1 ? g0 : (B.perm[1] == 1 ? g1 : g2);
        const int z = D == 2 ? 0 : (B.perm[0] == 2 ? g0 : (B.perm[1] == 2 ? g1 : g2));
        const int n = B.cn, bx = x / n, by = y / n, bz = D == 2 ? 0 : z / n;
        const int blk = B.bmap0[(bz * B.cnblk[1] + by) * B.cnblk[0] + bx];
        return blk * cells_of<D>(n) + cidx<D>(n, x - bx * n, y - by * n, z - bz * n);
    }
    // f - (L x - lambda x) in FP64 at a cell of level 0
    __device__ __forceinline__ double coarse_resid(const BotLev<T, D> &q, int a, int b, int p, const double *__restrict__ Wd0) const {
        const T *x = q.X + q.at(a, b, p);
        const double xc = (double)x[0];
        double s = 0;
#pragma unroll
        for (int i = 0; i < 3; i++) {
            if (D == 2 && i == 1) continue;
            const int st = i == 0 ? 1 : (i == 1 ? q.SA : q.SP), k = D == 2 && i == 2 ? 1 : i;
            const double lo = (double)x[-st] - xc, hi = (double)x[st] - xc;
            if (VAR) {
                const double *w = Wd0 + q.wat(a, b, p);
                s += w[(2 * k) * q.wn] * lo;
                s += w[(2 * k + 1) * q.wn] * hi;
            } else {
                s += L[0].inv_h2[B.perm[i]] * (lo + hi);
            }
        }
        return (double)q.F[q.fat(a, b, p)] - (s - P.helm * xc);
    }
    // sum of x over this CTA's cells of level 0, to every CTA (singular problems)
    __device__ __forceinline__ void coarse_sum(double wx) const {
        for (int o = 16; o > 0; o >>= 1) wx += __shfl_down_sync(0xffffffffu, wx, o);
        __shared__ double sh[kBotThreads / 32];
        if ((tid & 31) == 0) sh[tid >> 5] = wx;
        __syncthreads();
        if (tid == 0) {
            double sum = 0;
            for (int e = 0; e < (nth >> 5); e++) sum += sh[e];
            for (int k = 0; k < B.PB * B.PP; k++) st_cluster(rank_addr(part + rank, k), sum);
        }
    }
    // exact coarsest solve with the dense inverse: r in FP64, gathered by
    // every CTA, then each CTA applies the rows that belong to its cells
    __device__ void coarse_dense(const double *__restrict__ minv, const double *__restrict__ Wd0) const {
        const BotLev<T, D> q = lev(0);
        const unsigned mA = M[0].a, mB = M[0].b;
        const int cells = q.A * q.Bn * q.Pn, nrank = B.PB * B.PP;
        double wx = 0;
        for (int c = tid; c < cells; c += nth) {
            const int row = bot_div(c, mA), a = c - row * q.A, p = bot_div(row, mB), b = row - p * q.Bn;
            const double res = coarse_resid(q, a, b, p, Wd0);
            const int cr = coarse_row(a, q.gb + b, q.gp + p);
            for (int k = 0; k < nrank; k++) st_cluster(rank_addr(r + cr, k), res);
            wx += (double)q.X[q.at(a, b, p)];
        }
        if (B.singular) coarse_sum(wx);  // the border row: - sum V x
        cluster_sync();
        double border = 0;
        if (B.singular) {
            for (int k = 0; k < nrank; k++) border += part[k];
            border *= -L[0].vol;
        }
        // two rows per warp at a time: the residual is read once for them,
        // and their sums are reduced together
        const int lane = tid & 31, warp = tid >> 5, nw = nth >> 5;
        for (int c0 = 2 * warp; c0 < cells; c0 += 2 * nw) {
            const double *mr[2];
#pragma unroll
            for (int e = 0; e < 2; e++) {
                const int c = min(c0 + e, cells - 1);
                const int row = bot_div(c, mA), a = c - row * q.A, p = bot_div(row, mB), b = row - p * q.Bn;
                mr[e] = minv + (long long)coarse_row(a, q.gb + b, q.gp + p) * B.ns;
            }
            double acc[2] = {0, 0};
#pragma unroll 8
            for (int k = lane; k < B.nc; k += 32) {
                const double rk = r[k];
#pragma unroll
                for (int e = 0; e < 2; e++) acc[e] = fma(mr[e][k], rk, acc[e]);
            }
            const bool up = lane & 16;  // lanes 0-15 keep the first row, 16-31 the second
            double s = up ? acc[1] : acc[0];
            s += __shfl_xor_sync(0xffffffffu, up ? acc[0] : acc[1], 16);
            for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            const int c = c0 + (lane >> 4);
            if ((lane & 15) == 0 && c < cells) {
                if (B.singular) s = fma((lane ? mr[1] : mr[0])[B.nc], border, s);
                const int row = bot_div(c, mA), a = c - row * q.A, p = bot_div(row, mB), b = row - p * q.Bn;
                T *x = q.X + q.at(a, b, p);
                *x = (T)((double)*x + s);
            }
        }
        publish(q, q.X, -1);
    }
    // sum_k A(k) v(k) for k < n, by groups of G lanes of a warp (G a power of
    // two): every lane of the group returns it
    template <class Fa, class Fv> __device__ __forceinline__ static double dot(int n, int g, int G, Fa A, Fv v) {
        double s = 0;
#pragma unroll 4
        for (int k = g; k < n; k += G) s = fma(A(k), v(k), s);
        for (int o = 1; o < G; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        return s;
    }
    // Exact coarsest solve of the constant-coefficient operator by its
    // eigenvectors, which are products of one-dimensional ones:
    //   dx = Q_a Q_b G Q_b^T Q_a^T r,  G(ka, kb) = Q_p diag(1 / lambda) Q_p^T.
    // A + B + P FMAs per cell and direction instead of a row of the dense
    // inverse per cell (GB300 completes one FP64 instruction per SM in 16
    // cycles, and the inverse is 2 to 8 MB); the line between the two is drawn
    // where the layout is made.  Forward along a and b the CTA
    // works on its own planes of p and its own b (as kb), then every CTA
    // gathers the transform and solves its planes.
    __device__ void coarse_fd() const {
        const BotLev<T, D> q = lev(0);
        const int A = q.A, NB = q.NB, NP = B.n0[2], pl_ = q.Pn, bl_ = q.Bn;
        const int cells = A * bl_ * pl_;
        double *rr = r, *t1 = rr + B.mp * NB * A, *gg = t1 + B.mp * NB * A;  // [p][b][a] of own planes; gg: all planes
        double *u = rr, *v = t1;
        const double *qa = fd_tab, *qb = qa + A * A;  // [cell][mode], in shared memory
        double wx = 0;
        for (int c = tid; c < cells; c += nth) {
            const int row = bot_div(c, M[0].a), a = c - row * A, p = bot_div(row, M[0].b), b = row - p * bl_;
            const double res = coarse_resid(q, a, b, p, nullptr);
            for (int k = 0; k < B.PB; k++) st_cluster(rank_addr(rr + (p * NB + q.gb + b) * A + a, rank / B.PB * B.PB + k), res);
            wx += (double)q.X[q.at(a, b, p)];
        }
        if (B.singular) coarse_sum(wx);
        cluster_sync();
        // lanes per sum: long sums are cut (a chain of FP64 FMAs takes 64 cycles each)
        const int ga = A >= 16 ? 4 : 1, gb = NB >= 16 ? 4 : 1, gp = NP >= 16 ? 4 : 1;
        auto each = [&](int n, int G, auto &&body) {  // body(item, lane in group) for every item; a warp past the last one stops
            const int per = nth / G;
            for (int o0 = 0; o0 + (tid & ~31) / G < n; o0 += per) body(o0 + tid / G, tid & (G - 1));
        };
        each(pl_ * NB * A, ga, [&](int o, int g) {  // along a, every b of the own planes
            const int oc = min(o, pl_ * NB * A - 1), row = bot_div(oc, M[0].a), ka = oc - row * A;
            const double s = dot(A, g, ga, [&](int k) { return qa[k * A + ka]; }, [&](int k) { return rr[row * A + k]; });
            if (g == 0 && o == oc) t1[oc] = s;
        });
        __syncthreads();
        each(cells, D == 3 ? gb : 1, [&](int o, int g) {  // along b, own kb; to every CTA
            const int oc = min(o, cells - 1), row = bot_div(oc, M[0].a), ka = oc - row * A;
            const int p = bot_div(row, M[0].b), kb = q.gb + row - p * bl_;
            double s;
            if (D == 3) s = dot(NB, g, gb, [&](int k) { return qb[k * NB + kb]; }, [&](int k) { return t1[(p * NB + k) * A + ka]; });
            else s = t1[oc];
            if (g == 0 && o == oc)
                for (int k = 0; k < B.PB * B.PP; k++) st_cluster(rank_addr(gg + ((q.gp + p) * NB + kb) * A + ka, k), s);
        });
        cluster_sync();
        const int plane = NB * A;
        each(pl_ * plane, gp, [&](int o, int g) {  // the solve along p, at the own planes
            const int oc = min(o, pl_ * plane - 1), p = oc / plane, k0 = oc - p * plane;
            const double *G = fd_g + (long long)(q.gp + p) * NP * plane + k0;
            const double s = dot(NP, g, gp, [&](int k) { return G[(long long)k * plane]; }, [&](int k) { return gg[k * plane + k0]; });
            if (g == 0 && o == oc) u[oc] = s;
        });
        __syncthreads();
        if (D == 3) {
            each(cells, gb, [&](int o, int g) {  // back along b, own b
                const int oc = min(o, cells - 1), row = bot_div(oc, M[0].a), ka = oc - row * A;
                const int p = bot_div(row, M[0].b), b = row - p * bl_;
                const double s = dot(NB, g, gb, [&](int k) { return qb[(q.gb + b) * NB + k]; },
                                     [&](int k) { return u[(p * NB + k) * A + ka]; });
                if (g == 0 && o == oc) v[oc] = s;
            });
            __syncthreads();
        }
        double mean = 0;
        if (B.singular) {  // the constants: x + dx has zero mean
            for (int k = 0; k < B.PB * B.PP; k++) mean += part[k];
            mean /= B.nc;
        }
        const double *vv = D == 3 ? v : u;
        each(cells, ga, [&](int o, int g) {
            const int oc = min(o, cells - 1), row = bot_div(oc, M[0].a), a = oc - row * A;
            const int p = bot_div(row, M[0].b), b = row - p * bl_;
            const double s = dot(A, g, ga, [&](int k) { return qa[a * A + k]; }, [&](int k) { return vv[row * A + k]; });
            if (g == 0 && o == oc) {
                T *x = q.X + q.at(a, b, p);
                *x = (T)((double)*x + (s - mean));
            }
        });
        publish(q, q.X, -1);
    }
    __device__ __forceinline__ void coarse(const double *minv, const double *Wd0) const {
        if (!VAR && B.fd) coarse_fd();
        else coarse_dense(minv, Wd0);
    }
    __device__ void vcycle(int top, const double *minv, const double *Wd0) const {
        for (int l = top; l >= 1; l--) {
            smooth(l, B.dn[l]);
            restrict_to(l);
        }
        coarse(minv, Wd0);
        for (int l = 1; l <= top; l++) {
            prolong_to(l);
            smooth(l, B.up[l]);
        }
    }
    // A run of VW cells along a on the top level: local coordinates of the
    // first, its in-block x, y, z, its block and its cell in the block.
    struct Where {
        int a, b, p, x, y, z, blk, cell;
    };
    template <int VW> __device__ __forceinline__ Where where(const BotLev<T, D> &q, int c, unsigned mA, unsigned mB, unsigned mN) const {
        Where w;
        const int row = bot_div(c, mA), ra = q.A / VW;
        w.a = (c - row * ra) * VW;
        w.p = bot_div(row, mB);
        w.b = row - w.p * q.Bn;
        const int g1 = q.gb + w.b, g2 = q.gp + w.p, n = B.n;
        const int x = B.perm[0] == 0 ? w.a : (B.perm[1] == 0 ? g1 : g2);
        const int y = B.perm[0] == 1 ? w.a : (B.perm[1] == 1 ? g1 : g2);
        const int z = D == 2 ? 0 : (B.perm[0] == 2 ? w.a : (B.perm[1] == 2 ? g1 : g2));
        const int bx = bot_div(x, mN), by = bot_div(y, mN), bz = D == 2 ? 0 : bot_div(z, mN);
        w.x = x - bx * n;
        w.y = y - by * n;
        w.z = z - bz * n;
        w.blk = bmap[(bz * B.nblk[1] + by) * B.nblk[0] + bx];
        w.cell = cidx<D>(n, w.x, w.y, w.z);
        return w;
    }
    template <int VW> struct Run {
        T v[VW];
    };
    template <int VW> __device__ __forceinline__ static Run<VW> ldrun(const T *p) {
        Run<VW> r;
        if constexpr (VW == 4 && sizeof(T) == 4) {
            const float4 t = *reinterpret_cast<const float4 *>(p);
            r.v[0] = t.x; r.v[1] = t.y; r.v[2] = t.z; r.v[3] = t.w;
        } else if constexpr (VW == 4) {
            const double2 t = reinterpret_cast<const double2 *>(p)[0], u = reinterpret_cast<const double2 *>(p)[1];
            r.v[0] = t.x; r.v[1] = t.y; r.v[2] = u.x; r.v[3] = u.y;
        } else {
            r.v[0] = *p;
        }
        return r;
    }
    template <int VW> __device__ __forceinline__ static void strun(T *p, const Run<VW> &r) {
        if constexpr (VW == 4 && sizeof(T) == 4) {
            *reinterpret_cast<float4 *>(p) = make_float4(r.v[0], r.v[1], r.v[2], r.v[3]);
        } else if constexpr (VW == 4) {
            reinterpret_cast<double2 *>(p)[0] = make_double2(r.v[0], r.v[1]);
            reinterpret_cast<double2 *>(p)[1] = make_double2(r.v[2], r.v[3]);
        } else {
            *p = r.v[0];
        }
    }
    // the VW cells at padded offset i
    template <int VW> __device__ __forceinline__ static Run<VW> pick(const T *x) {
        Run<VW> r;
#pragma unroll
        for (int e = 0; e < VW; e++) r.v[e] = x[e];
        return r;
    }
    // the block-face ghosts beside a run of the top level, from the padded slab, to the ghost array Y
    template <int VW> __device__ __forceinline__ void ghosts_out(const BotLev<T, D> &q, const Where &w, T *__restrict__ Y) const {
        const int n = B.n, F = face_of<D>(n);
        const long long g0 = B.ghost_first + (long long)w.blk * (2 * D * F);
        const T *x = q.X + q.at(w.a, w.b, w.p);
#pragma unroll
        for (int d = 0; d < D; d++) {
            const int st = B.perm[0] == d ? 1 : (B.perm[1] == d ? q.SA : q.SP), in = d == 0 ? w.x : (d == 1 ? w.y : w.z);
            const int u = tidx<D>(n, d, w.x, w.y, w.z);
            if (VW == 4 && d == 0) {  // the run lies along x: at most one cell at each end
                if (in == 0) Y[g0 + u] = x[-1];
                if (in + 4 == n) Y[g0 + F + u] = x[4];
                continue;
            }
            if (in == 0) strun<VW>(Y + g0 + (2 * d) * F + u, pick<VW>(x - st));
            if (in == n - 1) strun<VW>(Y + g0 + (2 * d + 1) * F + u, pick<VW>(x + st));
        }
    }
    template <int VW> __device__ __forceinline__ void load_top() const {
        const BotLev<T, D> q = lev(B.top);
        const unsigned mA = VW == 4 ? M[B.top].qa : M[B.top].a, mB = M[B.top].b, mN = bot_magic(B.n);
        const int runs = q.A / VW * q.Bn * q.Pn, C = cells_of<D>(B.n);
        constexpr int kBatch = 4;  // runs in flight per thread
        for (int c0 = tid; c0 < runs; c0 += kBatch * nth) {
            Where w[kBatch];
            Run<VW> x[kBatch], f[kBatch];
#pragma unroll
            for (int e = 0; e < kBatch; e++) w[e] = where<VW>(q, min(c0 + e * nth, runs - 1), mA, mB, mN);
#pragma unroll
            for (int e = 0; e < kBatch; e++) {
                const long long o = B.cell_first + (long long)w[e].blk * C + w[e].cell;
                x[e] = ldrun<VW>(G.X + o);
                f[e] = ldrun<VW>(G.F + o);
            }
#pragma unroll
            for (int e = 0; e < kBatch; e++) {
                if (c0 + e * nth >= runs) continue;
                const int i = q.at(w[e].a, w[e].b, w[e].p);  // padded rows: element stores
#pragma unroll
                for (int k = 0; k < VW; k++) {
                    q.X[i + k] = x[e].v[k];
                    q.F[i - q.SP + k] = f[e].v[k];
                }
            }
        }
        publish(q, q.X, -1);
        if (B.nref == 0) return;
        // blocks covered by a finer level: f += L x, and v_old for the prolongation to it
        const T w0 = ih(B.top, 0), w1 = ih(B.top, 1), w2 = ih(B.top, 2);
        for (int c = tid; c < runs; c += nth) {
            const Where w = where<VW>(q, c, mA, mB, mN);
            if (w.blk >= B.nref) continue;
#pragma unroll
            for (int k = 0; k < VW; k++) q.F[q.fat(w.a + k, w.b, w.p)] += lap(q, w.a + k, w.b, w.p, w0, w1, w2);
            strun<VW>(G.V + B.cell_first + (long long)w.blk * C + w.cell, pick<VW>(q.X + q.at(w.a, w.b, w.p)));
            ghosts_out<VW>(q, w, G.VG);
        }
        cluster_sync();  // halos are read above and change below
    }
    template <int VW> __device__ __forceinline__ void store_top() const {
        const BotLev<T, D> q = lev(B.top);
        const unsigned mA = VW == 4 ? M[B.top].qa : M[B.top].a, mB = M[B.top].b, mN = bot_magic(B.n);
        const int runs = q.A / VW * q.Bn * q.Pn, C = cells_of<D>(B.n);
        for (int c = tid; c < runs; c += nth) {
            const Where w = where<VW>(q, c, mA, mB, mN);
            strun<VW>(G.X + B.cell_first + (long long)w.blk * C + w.cell, pick<VW>(q.X + q.at(w.a, w.b, w.p)));
            ghosts_out<VW>(q, w, G.XG);
        }
    }
};

template <class T, int D, bool VAR>
__global__ void __launch_bounds__(kBotThreads, 1)
k_bottom(KParams P, Fields<T> F, const __grid_constant__ BotPlan B, const double *__restrict__ minv,
         const T *__restrict__ Wd, const double *__restrict__ Wd0, T omega) {
    extern __shared__ __align__(16) unsigned char bot_smem[];
    __shared__ __align__(16) LevelDesc sL[kBotMaxLev];
    __shared__ BotMagic sM[kBotMaxLev];
    __shared__ int s_map[kBotMap];
    const int rank = (int)cluster_rank(), tid = threadIdx.x, nth = blockDim.x;
    for (int i = tid; i < (int)(sizeof(LevelDesc) / 4) * (B.top + 1); i += nth)
        reinterpret_cast<int *>(sL)[i] = reinterpret_cast<const int *>(P.L)[i];
    const int nmap = B.nblk[0] * B.nblk[1] * B.nblk[2];
    if (nmap <= kBotMap)
        for (int i = tid; i < nmap; i += nth) s_map[i] = B.bmap[i];
    const int pb = rank % B.PB, pp = rank / B.PB;
    auto cut = [](int k, int n, int parts) { return (int)((long long)k * n / parts); };
    const int b0 = cut(pb, B.n0[1], B.PB), b1 = cut(pb + 1, B.n0[1], B.PB);
    const int p0 = cut(pp, B.n0[2], B.PP), p1 = cut(pp + 1, B.n0[2], B.PP);
    if (tid <= B.top) {
        const int A = B.n0[0] << tid, Bn = D == 3 ? (b1 - b0) << tid : 1;
        sM[tid] = BotMagic{bot_magic(A), bot_magic(max(1, A >> 1)), bot_magic(max(1, A >> 2)), bot_magic(Bn),
                           bot_magic(max(1, Bn >> 1)), bot_magic(max(1, A >> 5))};
    }
    const bool perb = D == 3 && P.bct[2 * B.perm[1]] == MG_BC_PERIODIC, perp = P.bct[2 * B.perm[2]] == MG_BC_PERIODIC;
    const int pbl = pb > 0 ? pb - 1 : (perb ? B.PB - 1 : -1), pbh = pb < B.PB - 1 ? pb + 1 : (perb ? 0 : -1);
    const int ppl = pp > 0 ? pp - 1 : (perp ? B.PP - 1 : -1), pph = pp < B.PP - 1 ? pp + 1 : (perp ? 0 : -1);
    double *part = reinterpret_cast<double *>(bot_smem), *tab = part + 16;
    const int ntab = !VAR && B.fd ? B.n0[0] * B.n0[0] + (D == 3 ? B.n0[1] * B.n0[1] : 0) : 0;
    for (int i = tid; i < ntab; i += nth) tab[i] = B.fdtab[i];
    Bottom<T, D, VAR> K{P, B, F, Wd, sL, sM, reinterpret_cast<T *>(bot_smem + B.array0), part, tab + ntab, tab,
                        B.fdtab + ntab, tid, nth, rank,
                        b0, b1 - b0, p0, p1 - p0,
                        pbl < 0 ? 0 : cut(pbl + 1, B.n0[1], B.PB) - cut(pbl, B.n0[1], B.PB),
                        ppl < 0 ? 0 : cut(ppl + 1, B.n0[2], B.PP) - cut(ppl, B.n0[2], B.PP),
                        pbl < 0 ? -1 : pp * B.PB + pbl, pbh < 0 ? -1 : pp * B.PB + pbh,
                        ppl < 0 ? -1 : ppl * B.PB + pb, pph < 0 ? -1 : pph * B.PB + pb,
                        P.bct[2 * B.perm[0]] == MG_BC_PERIODIC, omega, nmap <= kBotMap ? (const int *)s_map : B.bmap};
    __syncthreads();
    cluster_sync();  // every CTA has started: its shared memory may be written
    // rows of 4 cells where a runs along x and blocks hold whole rows of 4
    // (offsets are then multiples of 4 elements), else cell by cell
    const bool vec = B.perm[0] == 0 && (B.n & 3) == 0;
    if (vec) K.template load_top<4>();
    else K.template load_top<1>();
    if (B.fmg) {
        for (int l = B.top; l >= 1; l--) K.restrict_to(l);
        K.coarse(minv, Wd0);
        for (int l = 1; l <= B.top; l++) {
            K.prolong_to(l);
            K.vcycle(l, minv, Wd0);
        }
    } else {
        K.vcycle(B.top, minv, Wd0);
    }
    if (vec) K.template store_top<4>();
    else K.template store_top<1>();
}

// Coefficients of one complete level in the dense order of the cluster
// kernel, [slot][p][b][a]: the 2D face weights in local face order and the
// reciprocal diagonal, from the block-ordered FP64 table.
template <class T, int D>
__global__ void __launch_bounds__(256) k_bottom_coef(BotPlan B, int l, const int *__restrict__ bmap, int n, int nbx,
                                                     int nby, long long cell_first, const double *__restrict__ W,
                                                     T *__restrict__ out) {
    pdl_entry();
    const int A = B.n0[0] << l, NB = D == 3 ? B.n0[1] << l : 1, NP = B.n0[2] << l, C = cells_of<D>(n);
    const long long cells = (long long)A * NB * NP;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < cells; c += (long long)gridDim.x * blockDim.x) {
        const int g0 = (int)(c % A), g1 = (int)(c / A % NB), g2 = (int)(c / ((long long)A * NB));
        const int x = B.perm[0] == 0 ? g0 : (B.perm[1] == 0 ? g1 : g2);
        const int y = B.perm[0] == 1 ? g0 : (B.perm[1] == 1 ? g1 : g2);
        const int z = D == 2 ? 0 : (B.perm[0] == 2 ? g0 : (B.perm[1] == 2 ? g1 : g2));
        const int blk = bmap[(z / n * nby + y / n) * nbx + x / n];
        const double *w = W + (cell_first + (long long)blk * C) * wstride(D) + cidx<D>(n, x % n, y % n, z % n);
        int slot = 0;
        for (int i = 0; i < 3; i++) {
            if (D == 2 && i == 1) continue;
            for (int s = 0; s < 2; s++) out[cells * slot++ + c] = (T)w[(2 * B.perm[i] + s) * C];
        }
        out[cells * slot + c] = (T)w[(2 * D + 1) * C];
    }
}

// The inverses along p of the eigenvector solve, [p'][p][kb][ka]: one sum over
// the NP modes per value.  On the device because the sums are plane NP^3: 32 s
// on one host core for a coarsest level of 3 x 1800 cells.
__global__ void __launch_bounds__(256) k_fd_table(const double *__restrict__ Q, const double *__restrict__ w, int plane,
                                                  int NP, double *__restrict__ out) {
    pdl_entry();
    const long long total = (long long)plane * NP * NP;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total; e += (long long)gridDim.x * blockDim.x) {
        const int kab = (int)(e % plane), s = (int)(e / plane % NP), p = (int)(e / plane / NP);
        double v = 0;
        for (int k = 0; k < NP; k++)
            v = fma(Q[(long long)k * NP + p] * w[(long long)k * plane + kab], Q[(long long)k * NP + s], v);
        out[e] = v;
    }
}

// ------------------------------------------------------------ host side ---

template <class T, int D, bool VAR> static int bot_clusters(int cs, size_t smem) {
    auto kern = k_bottom<T, D, VAR>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBotSmem) != cudaSuccess ||
        (cs > 8 && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)) {
        cudaGetLastError();
        return 0;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)cs);
    cfg.blockDim = dim3(kBotThreads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim = {(unsigned)cs, 1, 1};
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}
template <class T> static int bot_clusters_of(const mg_tree *t, int cs, size_t smem) {
    if (t->dim == 2) return t->var_eps ? bot_clusters<T, 2, true>(cs, smem) : bot_clusters<T, 2, false>(cs, smem);
    return t->var_eps ? bot_clusters<T, 3, true>(cs, smem) : bot_clusters<T, 3, false>(cs, smem);
}

// Shared-memory layout for levels 0 .. top on PB x PP CTAs; bytes needed, 0 if the slabs do not exist.
template <class T> static size_t bot_layout(const mg_tree *t, BotPlan &B, int top, bool jac) {
    const int D = t->dim;
    B.mb = (B.n0[1] + B.PB - 1) / B.PB;
    B.mp = (B.n0[2] + B.PP - 1) / B.PP;
    const long long tab = (long long)B.n0[0] * B.n0[0] + (D == 3 ? (long long)B.n0[1] * B.n0[1] : 0);
    // by eigenvectors from 400 cells on: 7.7 against 26 us for 36 x 27 cells,
    // 13 against 14 for 8^3; below, its five dependent FP64 stages take longer
    // than the rows of the inverse (8.0 against 6.1 for 180 cells, 5.6 against
    // 3.7 for 8 x 8).  Nothing between 180 and 512 cells was measured.
    B.fd = !t->var_eps && t->nc >= 400 && tab <= 2600;
    // The coarsest solve reads the inverse (nc^2 values) or the tables along p
    // (nc n_p) through 16 SMs.  Above 2048^2 values that takes longer than the
    // whole chip needs, launches and all, for every level of the cycle: 4
    // V-cycles with a dense inverse of 1800 cells 461 against 526 us, 2520
    // 833 / 790, 3348 1063 / 765, 5400 2250 / 1016; with tables of 3500 x 70
    // values 312 / 585, of 5400 x 1800 1094 / 742.
    if ((long long)t->nc * (B.fd ? B.n0[2] : t->nc) > 2048LL * 2048) return 0;
    const long long plane = (long long)B.n0[0] * (D == 3 ? B.n0[1] : 1);
    const long long scratch = B.fd ? tab + (2 * B.mp + B.n0[2]) * plane : t->ns;
    const size_t head = sizeof(double) * (size_t)(16 + scratch);
    if (head > kBotSmem) return 0;
    B.array0 = (int)((head + 15) / 16 * 16);
    long long o = 0;
    auto take = [&](long long n) { const long long at = o; o += (n + 3) / 4 * 4; return (int)at; };
    for (int l = 0; l <= top; l++) {
        const long long A = (long long)B.n0[0] << l, Bn = D == 3 ? (long long)B.mb << l : 1, Pn = (long long)B.mp << l;
        const long long sp = (A + 2) * (D == 3 ? Bn + 2 : 1);
        if (l > 0 && (A / 2 * Bn * Pn + kBotThreads - 1) / kBotThreads > kBotPer) return 0;
        B.offx[l] = take(sp * (Pn + 2));
        B.offf[l] = take(sp * Pn);
        B.offv[l] = l < top ? take(sp * (Pn + 2)) : 0;
        if (l == top) B.offj = jac ? take(sp * (Pn + 2)) : 0;
        if (B.array0 + o * (long long)sizeof(T) > (long long)kBotSmem) return 0;
    }
    B.top = top;
    return B.array0 + (size_t)o * sizeof(T);
}

// The cut of the cluster for one CTA count: which dimension stays whole and
// how the others are split, by the largest slab.
static bool bot_cut(const mg_tree *t, BotPlan &B, int cs) {
    const int *nc = t->lev[0].ncell;
    long long best = -1;
    BotPlan w = B;
    static const int order3[6][3] = {{0, 1, 2}, {0, 2, 1}, {1, 0, 2}, {1, 2, 0}, {2, 0, 1}, {2, 1, 0}};
    static const int order2[2][3] = {{0, 2, 1}, {1, 2, 0}};
    const int no = t->dim == 3 ? 6 : 2;
    for (int o = 0; o < no; o++) {
        const int *pm = t->dim == 3 ? order3[o] : order2[o];
        for (int pb = 1; pb <= (t->dim == 3 ? cs : 1); pb++) {
            if (cs % pb) continue;
            const int pp = cs / pb, n1 = t->dim == 3 ? nc[pm[1]] : 1, n2 = nc[pm[2]];
            if (pb > n1 || pp > n2) continue;
            const long long mb = (n1 + pb - 1) / pb, mp = (n2 + pp - 1) / pp;
            // largest slab, with its halo (the pushes and the padded copies)
            const long long cost = (long long)nc[pm[0]] * (4 * mb * mp + (pb > 1 ? 2 * mp : 0) + (pp > 1 ? 2 * mb : 0));
            if (best >= 0 && cost >= best) continue;
            best = cost;
            for (int e = 0; e < 3; e++) w.perm[e] = pm[e];
            w.n0[0] = nc[pm[0]];
            w.n0[1] = n1;
            w.n0[2] = n2;
            w.PB = pb;
            w.PP = pp;
        }
    }
    if (best < 0) return false;
    B = w;
    return true;
}

// Orthonormal eigenvectors (column k: mode k) and eigenvalues of minus the
// second difference of n cell-centred values, with the ghost rules of Sec. 2.6
// at the two ends (Dirichlet -x, Neumann and axis x, or periodic).
static void line_modes(int n, double h, int lo, int hi, std::vector<double> &Q, std::vector<double> &lam) {
    Q.assign((size_t)n * n, 0.0);
    lam.assign(n, 0.0);
    const bool dl = lo == MG_BC_DIRICHLET, dh = hi == MG_BC_DIRICHLET;
    for (int k = 0; k < n; k++) {
        double th;
        bool sine;
        if (lo == MG_BC_PERIODIC) {
            const int m = (k + 1) / 2;
            th = 2.0 * M_PI * m / n;
            sine = k > 0 && k % 2 == 0;
        } else if (dl == dh) {
            th = M_PI * (dl ? k + 1 : k) / n;
            sine = dl;
        } else {
            th = M_PI * (k + 0.5) / n;
            sine = dl;
        }
        lam[k] = (2.0 - 2.0 * std::cos(th)) / (h * h);
        double s2 = 0;
        for (int i = 0; i < n; i++) {
            const double at = lo == MG_BC_PERIODIC ? th * i : th * (i + 0.5);
            const double v = sine ? std::sin(at) : std::cos(at);
            Q[(size_t)i * n + k] = v;
            s2 += v * v;
        }
        for (int i = 0; i < n; i++) Q[(size_t)i * n + k] /= std::sqrt(s2);
    }
}

// Tables of the eigenvector solve of the coarsest level (coarse_fd) into
// S.d_fd: the modes along a and b, then per (ka, kb) the inverse along p,
// Q_p diag(-1 / (lam_a + lam_b + lam_p + lambda)) Q_p^T, as [p'][p][kb][ka].
// The constants of a singular problem get 0.  False: no memory.
static bool fd_tables(mg_tree *t, const BotPlan &B, BotState &S) {
    const LevelHost &L = t->lev[0];
    std::vector<double> Q[3], lam[3];
    for (int i = 0; i < 3; i++) {
        const int d = B.perm[i];
        if (t->dim == 2 && i == 1) {
            Q[1] = {1.0};
            lam[1] = {0.0};
            continue;
        }
        line_modes(L.ncell[d], L.h[d], t->bc.type[2 * d], t->bc.type[2 * d + 1], Q[i], lam[i]);
    }
    std::vector<double> head(Q[0]);
    if (t->dim == 3) head.insert(head.end(), Q[1].begin(), Q[1].end());
    const size_t A = B.n0[0], NB = t->dim == 3 ? B.n0[1] : 1, NP = B.n0[2], plane = A * NB;
    // the sums along p run on the device: modes [k][p], then weights [k][kb][ka]
    std::vector<double> in(NP * NP + NP * plane);
    for (size_t k = 0; k < NP; k++) {
        for (size_t p = 0; p < NP; p++) in[k * NP + p] = Q[2][p * NP + k];
        for (size_t kb = 0; kb < NB; kb++)
            for (size_t ka = 0; ka < A; ka++) {
                const bool constant = t->singular && ka == 0 && kb == 0 && k == 0;
                in[NP * NP + (k * NB + kb) * A + ka] = constant ? 0.0 : -1.0 / (lam[0][ka] + lam[1][kb] + lam[2][k] + t->helm);
            }
    }
    const size_t total = plane * NP * NP;
    double *d_in = nullptr;
    bool ok = cudaMalloc((void **)&S.d_fd, sizeof(double) * (head.size() + total)) == cudaSuccess &&
              cudaMalloc((void **)&d_in, sizeof(double) * in.size()) == cudaSuccess &&
              upload(S.d_fd, head.data(), sizeof(double) * head.size(), t->stream) == cudaSuccess &&
              upload(d_in, in.data(), sizeof(double) * in.size(), t->stream) == cudaSuccess;
    if (ok) {
        ++t->launches;
        launch_k(k_fd_table, (int)std::min<size_t>((total + 255) / 256, 32 * (size_t)t->nsm), 256, 0, t->stream,
                 (const double *)d_in, (const double *)(d_in + NP * NP), (int)plane, (int)NP, S.d_fd + head.size());
        ok = cudaStreamSynchronize(t->stream) == cudaSuccess;
    }
    cudaFree(d_in);
    if (!ok) cudaGetLastError();
    return ok;
}

template <class T> static void bot_plan(mg_tree *t, bool jac, BotState &S) {
    S.tried = true;
    S.plan.top = 0;
    if (t->is_batch || t->geom != MG_CART || t->lev.size() < 2) return;
    int base = 0;  // the base grid: the highest level that certainly covers the domain
    while (base + 1 < (int)t->lev.size() && t->lev[base].depth < 0) base++;
    // Above these sizes the whole chip beats 16 SMs.  Measured (16 CTAs,
    // whole solves, FP32 cycles in 3D): 32^3 as top level 10.9 ms, 64^3
    // 11.4 ms on the 19.8M-cell tree, launch by launch 11.4; 64 against 67
    // and 67 ms on the 256^3 variable-coefficient problem.  2D has smaller
    // faces: 62k cells 1.66 ms, 15k cells 1.81 ms, launch by launch 2.74.
    // FP64 32^3 against 16^3 as top level: 15.8 and 17.2 ms (128^3 Jacobi),
    // 7.4 and 9.7 ms (64^3 cleaning with its adjoint).  2D FP64 takes the 3D
    // limit unmeasured.
    const long long limit = sizeof(T) == 4 && t->dim == 2 ? 100000 : 40000;
    for (int cs : {16, 8, 4, 2, 1}) {
        BotPlan B{};
        if (!bot_cut(t, B, cs)) continue;
        for (int top = std::min(base, kBotMaxLev - 1); top >= 1; top--) {
            if (t->lev[top].ncells > limit) continue;
            BotPlan q = B;
            const size_t sm = bot_layout<T>(t, q, top, jac);
            if (!sm || sm > kBotSmem || bot_clusters_of<T>(t, cs, sm) < 1) continue;
            if (S.plan.top < top) {
                S.plan = q;
                S.smem = sm;
            }
            break;
        }
        if (S.plan.top > 0 && (S.plan.top == std::min(base, kBotMaxLev - 1) || cs <= 8)) break;
    }
    BotPlan &B = S.plan;
    if (B.top == 0) return;
    // block maps of levels 0 .. top: block coordinates -> index within the level
    std::vector<int> map;
    std::vector<long long> off;
    for (int l = 0; l <= B.top; l++) {
        const LevelHost &L = t->lev[l];
        off.push_back((long long)map.size());
        map.resize(map.size() + (size_t)L.nb);
        for (int b = 0; b < L.nb; b++) {
            const BlockDesc &q = t->blocks[L.first + b];
            map[off[l] + ((long long)q.ijk[2] * L.nblk[1] + q.ijk[1]) * L.nblk[0] + q.ijk[0]] = b;
        }
    }
    if (cudaMalloc((void **)&S.d_map, sizeof(int) * map.size()) != cudaSuccess ||
        upload(S.d_map, map.data(), sizeof(int) * map.size(), t->stream) != cudaSuccess) {
        cudaGetLastError();
        B.top = 0;
        return;
    }
    if (B.fd) {
        if (!fd_tables(t, B, S)) {
            B.top = 0;
            return;
        }
        B.fdtab = S.d_fd;
    }
    const LevelHost &L = t->lev[B.top], &L0 = t->lev[0];
    B.bmap = S.d_map + off[B.top];
    B.bmap0 = S.d_map + off[0];
    B.n = L.n;
    B.cn = L0.n;
    for (int d = 0; d < 3; d++) {
        B.nblk[d] = L.nblk[d];
        B.cnblk[d] = L0.nblk[d];
    }
    B.nref = L.nref;
    B.cell_first = L.cell_first;
    B.ghost_first = L.ghost_first;
    B.nc = t->nc;
    B.ns = t->ns;
    B.singular = t->singular ? 1 : 0;
    B.jac = jac ? 1 : 0;
    long long w = 0;
    for (int l = 0; l <= B.top; l++) {
        B.woff[l] = w;
        w += (2 * t->dim + 1) * t->lev[l].ncells;
    }
    S.wtotal = w;
    for (int l = 0; l <= B.top; l++) S.mapoff[l] = off[l];
}

template <class T> static void bot_coef_one(mg_tree *t, BotState &S, T *W, int top) {
    for (int l = 0; l <= top; l++) {
        const LevelHost &L = t->lev[l];
        ++t->launches;
        const int grid = (int)std::max<long long>(1, std::min<long long>((L.ncells + 255) / 256, 8LL * t->nsm));
        auto kern = t->dim == 2 ? k_bottom_coef<T, 2> : k_bottom_coef<T, 3>;
        launch_k(kern, grid, 256, 0, t->stream, S.plan, l, (const int *)S.d_map + S.mapoff[l], L.n, L.nblk[0], L.nblk[1],
                 L.cell_first, (const double *)t->d_wface, W + S.plan.woff[l]);
    }
}

// The level the cluster kernel runs from (0: none) for precision T and the
// current smoother, as bottom_prepare left it (cycles are enqueued inside
// stream captures, so nothing is built here).
template <class T> int bottom_level(mg_tree *t) {
    const int prec = sizeof(T) == 4 ? 1 : 0;
    if (!t->bottom_on || t->tail_cells > 0 || t->coarse_mode != MG_COARSE_EXACT) return 0;
    const BotState &S = t->bottom[prec][t->smoother == MG_SMOOTH_JACOBI ? 1 : 0];
    for (int l = 0; l <= S.plan.top && l < (int)t->pinned[prec].size(); l++)
        if (t->pinned[prec][l]) return 0;  // a pinned level runs its own sweeps
    return t->var_eps && !S.d_w ? 0 : S.plan.top;
}

// Builds the plan of the current smoother and, with variable eps, its dense
// coefficients, where missing.  Without them the cycle runs launch by launch.
template <class T> void bottom_prepare(mg_tree *t) {
    const bool jac = t->smoother == MG_SMOOTH_JACOBI;
    BotState &S = t->bottom[sizeof(T) == 4 ? 1 : 0][jac ? 1 : 0];
    if (!S.tried) bot_plan<T>(t, jac, S);
    if (S.plan.top == 0 || !t->var_eps || S.d_w) return;
    if (cudaMalloc(&S.d_w, sizeof(T) * (size_t)S.wtotal) != cudaSuccess ||
        cudaMalloc((void **)&S.d_w0, sizeof(double) * (size_t)(2 * t->dim + 1) * t->lev[0].ncells) != cudaSuccess) {
        cudaGetLastError();
        cudaFree(S.d_w);
        S.d_w = nullptr;
        return;
    }
    bot_coef_one<T>(t, S, (T *)S.d_w, S.plan.top);
    bot_coef_one<double>(t, S, S.d_w0, 0);
}

// dense coefficients of the existing plans after a change of eps
void bottom_coef(mg_tree *t) {
    for (int prec = 0; prec < 2; prec++)
        for (int jac = 0; jac < 2; jac++) {
            BotState &S = t->bottom[prec][jac];
            if (!S.d_w) continue;
            if (prec) bot_coef_one<float>(t, S, (float *)S.d_w, S.plan.top);
            else bot_coef_one<double>(t, S, (double *)S.d_w, S.plan.top);
            bot_coef_one<double>(t, S, S.d_w0, 0);
        }
}

void bottom_free(mg_tree *t) {
    for (auto &p : t->bottom)
        for (BotState &S : p) {
            cudaFree(S.d_map);
            cudaFree(S.d_w);
            cudaFree(S.d_w0);
            cudaFree(S.d_fd);
            S = BotState();
        }
}

template <class T> void bottom_run(mg_tree *t, const KParams &P, Fields<T> &F, bool fmg, int nd, int nu) {
    const bool jac = t->smoother == MG_SMOOTH_JACOBI;
    const BotState &S = t->bottom[sizeof(T) == 4 ? 1 : 0][jac ? 1 : 0];
    BotPlan B = S.plan;
    B.fmg = fmg ? 1 : 0;
    for (int l = 0; l <= B.top; l++) {
        B.dn[l] = l < (int)t->sched_down.size() && t->sched_down[l] >= 0 ? t->sched_down[l] : nd;
        B.up[l] = l < (int)t->sched_up.size() && t->sched_up[l] >= 0 ? t->sched_up[l] : nu;
    }
    ++t->launches;
    auto go = [&](auto kern) {
        launch_cluster(kern, dim3((unsigned)(B.PB * B.PP)), dim3(kBotThreads), S.smem, t->stream, P, F, B,
                       (const double *)t->d_minv, (const T *)S.d_w, (const double *)S.d_w0, (T)t->omega);
    };
    if (t->dim == 2) t->var_eps ? go(k_bottom<T, 2, true>) : go(k_bottom<T, 2, false>);
    else t->var_eps ? go(k_bottom<T, 3, true>) : go(k_bottom<T, 3, false>);
}
template int bottom_level<double>(mg_tree *);
template int bottom_level<float>(mg_tree *);
template void bottom_prepare<double>(mg_tree *);
template void bottom_prepare<float>(mg_tree *);
template void bottom_run<double>(mg_tree *, const KParams &, Fields<double> &, bool, int, int);
template void bottom_run<float>(mg_tree *, const KParams &, Fields<float> &, bool, int, int);

}  // namespace mg
