// Multigrid levels worked by one thread-block cluster (sm_103a).
//
// The lower levels of the V-cycle are far too small to fill the GPU, and as
// one launch per half sweep they are a chain of dependent launches (1.2 us
// each); in a single CTA they are bound by that SM's issue rate and, in FP64,
// by its two FP64 FMAs per clock. Here a cluster of CTAs (up to 8 for a V-cycle,
// 16 for a whole solve) holds them in distributed shared memory: each CTA owns
// a slab of columns (an x range) of every level and works it with a wide margin
// of ghost columns. A cluster barrier takes 0.26-0.31 us (256-512 threads per
// CTA), a block barrier a quarter of that, so the ghosts are recomputed rather
// than exchanged: given the right-hand side on D ghost columns, each half sweep
// is valid on one column less, and a whole level (pre-smoothing, residual,
// prolongation, post-smoothing) passes with block barriers only. What crosses
// CTAs is the restricted right-hand side, once per level, stored into every CTA
// whose margin covers it (st.shared::cluster), followed by one cluster barrier.
// Slab boundaries are multiples of the x coarsening factor down to the
// coarsest level, so restriction stays inside a CTA.
//
// With E the columns beyond the slab on which a level's result is needed (the
// next finer level's prolongation), nu sweep pairs: the post-smoothing starts
// from colour-0 values valid E + 2 nu columns out, the pre-smoothing leaves
// them valid D - 2 (nu - 1) columns out, hence D = E + 4 nu - 2, and the next
// level's E is (E + 2 nu) / rx rounded up.
//
// The smoother, its order and the transfers are those of the per-level
// kernels (k_mg_rbgs, k_mg_resid_restrict): the same operations in the same
// order per cell. The coarsest level (at most kExactCells cells) is solved
// with its explicit inverse.
//
// Two kernels use it: k_mg_cluster, the V-cycle below a per-level hierarchy,
// and k_solve_cluster, a whole pressure solve of a small 2D grid (initial
// FP64 residual, PCG, defect correction) in one launch.
#pragma once
#include "oscar_kernels.cuh"

namespace oscar {

constexpr int kExactCells = 128;     // coarsest level solved exactly when at most this size
constexpr int kMaxCL = 16;           // levels of a cluster
constexpr int kMaxCluster = 16;      // CTAs of a cluster (above 8 needs the non-portable attribute)
constexpr size_t kClSmemBytes = 220 * 1024;   // dynamic shared memory a CTA may use

// A level. The local index of cell (i, j, k) in a CTA whose slab starts at
// column s is (i - s + G) ps + j + ny k: columns are contiguous (ps >= ny nz,
// odd, so that both directions are free of bank conflicts).
template <typename M> struct ClLevel {
    int nx, ny, nz;          // global extents
    int sh;                  // log2 of the x coarsening from this level to the coarsest
    int rx, ry, rz;          // ratios to the next level (1 or 2)
    int nu;                  // sweep pairs per smoothing step
    int paired;              // neighbour terms of a direction are added to each other first
    int G, D, E;             // columns beyond the slab: held on each side, on which b is needed, on which x is needed
    int ncol, ps, nloc;      // local columns (widest slab), column stride, local cells
    int ce;                  // entries of a column in a colour list: ceil(ny / 2) nz
    float rncol, rny, rce;   // reciprocals for the cell decomposition
    const M *c[3], *idiag;
    // shared-memory byte offsets: reciprocal diagonal, low-face coefficients
    // per direction, colour lists (local indices by column), the coarse local
    // index of each colour-0 entry, slab starts of all ranks; x, b
    int oi, oc[3], ol[2], op, os;
    int ox, ob;
};
template <typename M> struct ClLevels {
    int n, nc, lnc;          // levels, CTAs (a power of two) and their log2
    int cols;                // columns of the coarsest level
    int img;                 // bytes of the image: what is fixed for a set of coefficients, at the start of shared memory
    int oinv, orow;          // in the image: the inverse's rows that the CTA works, and the local cell of each
    int ors, obx;            // residual scratch, gathered right-hand side of the coarsest level
    int ored;                // reduction scratch
    const M *inv;            // explicit inverse of the coarsest level (row-major)
    unsigned char *image;    // the images of all ranks, img bytes apart
    ClLevel<M> L[kMaxCL];
};

constexpr unsigned short kClNone = 0xFFFF;

__device__ __forceinline__ int cl_rank() {
    int r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// every thread of every CTA of the cluster arrives; shared-memory stores made
// before it (own and remote) are visible after it. A cluster of one CTA takes
// the block barrier.
__device__ __forceinline__ void cl_sync(int nc) {
    if (nc > 1) asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
    else __syncthreads();
}
__device__ __forceinline__ unsigned cl_addr(const void *p, int rank) {
    unsigned a = (unsigned)__cvta_generic_to_shared(p), r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void cl_store(unsigned a, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void cl_store(unsigned a, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}

// slab of rank r on a level: global columns [cl_start(r), cl_start(r + 1))
template <typename M> __host__ __device__ __forceinline__ int cl_start(const ClLevels<M> &P, const ClLevel<M> &L, int r) {
    const int s = ((r * P.cols) >> P.lnc) << L.sh;
    return s < L.nx ? s : L.nx;
}
// local columns [q0, q1) of the slab with d columns beyond it on each side, inside the domain
struct ClRange { int s, w, q0, q1; };
template <typename M>
__device__ __forceinline__ ClRange cl_range(const ClLevels<M> &P, const ClLevel<M> &L, int rank, int d) {
    ClRange r;
    r.s = cl_start(P, L, rank);
    r.w = cl_start(P, L, rank + 1) - r.s;
    r.q0 = L.G - min(min(d, L.G), r.s);
    r.q1 = min(L.G + r.w + min(d, L.G), L.G + L.nx - r.s);
    return r;
}
// columns beyond its slab on which a CTA works the coarsest level's solution
// itself: in FP64, bound by FP64 issue, none (the values are sent instead)
template <typename M> __host__ __device__ __forceinline__ int cl_exact_depth(const ClLevels<M> &P) {
    return sizeof(M) == sizeof(float) ? P.L[P.n - 1].E : 0;
}

// store v into field f (a shared-memory array in the level's layout) at global
// column i, position m of the column, in every other CTA whose ghosts of depth
// d cover it
template <typename M>
__device__ __forceinline__ void cl_push(const ClLevels<M> &P, const ClLevel<M> &L, unsigned char *sm, M *f, int i, int m,
                                        int d, int rank, M v) {
    const short *st = (const short *)(sm + L.os);
    for (int r = rank - 1; r >= 0; --r) {
        if (i >= st[r + 1] + d) break;
        cl_store(cl_addr(f + (i - st[r] + L.G) * L.ps + m, r), v);
    }
    for (int r = rank + 1; r < P.nc; ++r) {
        const int s = st[r];
        if (i < s - d) break;
        cl_store(cl_addr(f + (i - s + L.G) * L.ps + m, r), v);
    }
}

// idx / n and the remainder, without integer division (rn = 1 / n; exact below 2^22)
__device__ __forceinline__ int div_rem(int idx, int n, float rn, int &rem) {
    int q = (int)(((float)idx + 0.5f) * rn);
    rem = idx - q * n;
    if (rem < 0) { --q; rem += n; } else if (rem >= n) { ++q; rem -= n; }
    return q;
}

// The image of the cluster's levels, one per CTA of the cluster: coefficients
// and lists in the local layout, once per set of coefficients, so that every
// V-cycle (or solve) starts from one contiguous copy. Block (rank, slice).
constexpr int kPackSlices = 8, kPackThreads = 256;
template <int DIM, typename M>
__global__ void __launch_bounds__(kPackThreads) k_cl_pack(ClLevels<M> P, int *__restrict__ ctl) {
    griddep_wait();
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) ctl[C_PACK] += 1;   // set-ups of this step call
    const int rank = blockIdx.x, t = blockIdx.y * kPackThreads + threadIdx.x, nt = kPackSlices * kPackThreads;
    unsigned char *im = P.image + (size_t)rank * P.img;
    for (int l = 0; l < P.n; ++l) {
        const ClLevel<M> &L = P.L[l];
        const int s = cl_start(P, L, rank);
        M *id = (M *)(im + L.oi), *c0 = (M *)(im + L.oc[0]), *c1 = (M *)(im + L.oc[1]), *c2 = (M *)(im + L.oc[2]);
        for (int o = t; o < L.nloc; o += nt) {
            const int q = o / L.ps, m = o - q * L.ps, k = m / L.ny, j = m - k * L.ny, i = s - L.G + q;
            const bool in = i >= 0 && k < L.nz;
            M v0 = M(0), v1 = M(0), v2 = M(0), vi = M(0);
            if (in && i < L.nx) {
                const int gc = i + L.nx * (j + L.ny * k);
                v1 = L.c[1][i + L.nx * (j + (L.ny + 1) * k)];
                if (DIM == 3) v2 = L.c[2][gc];
                vi = L.idiag[gc];
            }
            if (in && i <= L.nx) v0 = L.c[0][i + (L.nx + 1) * (j + L.ny * k)];   // i = nx: the outlet, x = 0 beyond it
            id[o] = vi;
            c0[o] = v0;
            c1[o] = v1;
            if (DIM == 3) c2[o] = v2;
        }
        // colour lists: entry (column q, k, tj) holds the cell of that colour
        // among rows 2 tj and 2 tj + 1
        const int hj = (L.ny + 1) >> 1;
        const bool last = l + 1 == P.n;
        const ClLevel<M> &C = P.L[last ? l : l + 1];
        const int cs = cl_start(P, C, rank);
        for (int h = t; h < L.ncol * L.ce; h += nt) {
            const int q = h / L.ce, m = h - q * L.ce, k = m / hj, tj = m - k * hj;
            const int i = s - L.G + q;
#pragma unroll
            for (int colour = 0; colour < 2; ++colour) {
                const int j = 2 * tj + ((i + k + colour) & 1);
                const bool in = i >= 0 && i < L.nx && j < L.ny;
                ((unsigned short *)(im + L.ol[colour]))[h] = in ? (unsigned short)(q * L.ps + j + L.ny * k) : kClNone;
                if (colour == 0 && !last) {
                    const int qc = (i >> (L.rx >> 1)) - cs + C.G;
                    ((unsigned short *)(im + L.op))[h] =
                        in && qc >= 0 && qc < C.ncol ? (unsigned short)(qc * C.ps + (j >> (L.ry >> 1)) + C.ny * (k >> (L.rz >> 1)))
                                                     : (unsigned short)0;
                }
            }
        }
        for (int r = t; r <= P.nc; r += nt) ((short *)(im + L.os))[r] = (short)cl_start(P, L, r);
    }
    // rows of the coarsest level's inverse
    const ClLevel<M> &L = P.L[P.n - 1];
    const ClRange R = cl_range(P, L, rank, cl_exact_depth(P));
    const int ne = L.nx * L.ny * L.nz, pl = L.ny * L.nz, nr = (R.q1 - R.q0) * pl;
    M *inv = (M *)(im + P.oinv);
    for (int o = t; o < nr * ne; o += nt) {
        const int row = o / ne, q = row / pl, m = row - q * pl;
        inv[o] = P.inv[(size_t)(R.s - L.G + R.q0 + q + L.nx * m) * ne + o - row * ne];
    }
    for (int row = t; row < nr; row += nt) {
        const int q = row / pl, m = row - q * pl;
        ((unsigned short *)(im + P.orow))[row] = (unsigned short)((R.q0 + q) * L.ps + m);
    }
}

// start the copy of the CTA's image into shared memory; x and b cleared
// meanwhile. cp_async_wait_all and a barrier complete it.
template <typename M>
__device__ __forceinline__ void cl_load(const ClLevels<M> &P, unsigned char *sm, int rank) {
    const unsigned char *im = P.image + (size_t)rank * P.img;
    for (int q = threadIdx.x * 16; q < P.img; q += blockDim.x * 16) {
        const unsigned d = (unsigned)__cvta_generic_to_shared(sm + q);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(im + q) : "memory");
    }
    for (int l = 0; l < P.n; ++l) {
        const ClLevel<M> &L = P.L[l];
        M *x = (M *)(sm + L.ox), *b = (M *)(sm + L.ob);
        for (int c = threadIdx.x; c < L.nloc; c += blockDim.x) { x[c] = M(0); b[c] = M(0); }
    }
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// b + the sum of the neighbour terms of one row. FP32: one term after the
// other (the order of mg_row_sum), or the two of a direction first on the
// levels of at most cta_cells cells (paired): FP32 rounding in the V-cycle is
// amplified in the smoothest pressure mode, so a level's order is the same
// whichever cluster works it. FP64 is bound by FP64 issue: fused multiply-adds.
template <int DIM>
__device__ __forceinline__ float cl_row_sum(const float *w, const float *x, int c, int ps, int ny, bool paired, float b) {
    const float a0 = w[0] * x[c - ps], a1 = w[1] * x[c + ps];
    const float b0 = w[2] * x[c - 1], b1 = w[3] * x[c + 1];
    float off = a0 + a1;
    off = paired ? off + (b0 + b1) : (off + b0) + b1;
    if (DIM == 3) {
        const float d0 = w[4] * x[c - ny], d1 = w[5] * x[c + ny];
        off = paired ? off + (d0 + d1) : (off + d0) + d1;
    }
    return b + off;
}
template <int DIM>
__device__ __forceinline__ double cl_row_sum(const double *w, const double *x, int c, int ps, int ny, bool, double b) {
    double t = fma(w[0], x[c - ps], b);
    t = fma(w[1], x[c + ps], t);
    t = fma(w[2], x[c - 1], t);
    t = fma(w[3], x[c + 1], t);
    if (DIM == 3) {
        t = fma(w[4], x[c - ny], t);
        t = fma(w[5], x[c + ny], t);
    }
    return t;
}
template <int DIM>
__device__ __forceinline__ float cl_residual(const float *w, const float *x, int c, int ps, int ny, bool paired, float b) {
    float dg = 0.f;   // the diagonal as it was formed
#pragma unroll
    for (int a = 0; a < DIM; ++a) dg += w[2 * a] + w[2 * a + 1];
    return b - (dg * x[c] - cl_row_sum<DIM>(w, x, c, ps, ny, paired, 0.f));
}
template <int DIM>
__device__ __forceinline__ double cl_residual(const double *w, const double *x, int c, int ps, int ny, bool paired, double b) {
    double dg = 0.0;
#pragma unroll
    for (int a = 0; a < DIM; ++a) dg += w[2 * a] + w[2 * a + 1];
    return fma(-dg, x[c], cl_row_sum<DIM>(w, x, c, ps, ny, paired, b));
}
// the coefficients of a row, from the low faces of the cell and its high neighbours
template <int DIM, typename M>
__device__ __forceinline__ void cl_row(const ClLevel<M> &L, unsigned char *sm, int c, M *w) {
    const M *c0 = (const M *)(sm + L.oc[0]), *c1 = (const M *)(sm + L.oc[1]), *c2 = (const M *)(sm + L.oc[2]);
    w[0] = c0[c];
    w[1] = c0[c + L.ps];
    w[2] = c1[c];
    w[3] = c1[c + 1];
    if (DIM == 3) {
        w[4] = c2[c];
        w[5] = c2[c + L.ny];
    }
}

// A thread's cells of a level, K list entries of each colour with their rows
// in registers: loaded once for the half sweeps of a smoothing step, which
// then read only x from shared memory. K = 0: any number of entries, the rows
// read again in every half sweep.
template <int DIM, typename M, int K> struct ClCells {
    int c[2][K], dist[2][K];   // local cell; columns outside the slab (a large number: no cell)
    M w[2][K][2 * DIM], id[2][K], b[2][K];
    __device__ __forceinline__ void load(const ClLevels<M> &P, const ClLevel<M> &L, unsigned char *sm, int rank) {
        const ClRange R = cl_range(P, L, rank, L.D);
        const M *bs = (const M *)(sm + L.ob), *ids = (const M *)(sm + L.oi);
#pragma unroll
        for (int u = 0; u < K; ++u) {
            const int h = R.q0 * L.ce + threadIdx.x + u * blockDim.x;
            const bool in = h < R.q1 * L.ce;
            int rem;
            const int q = div_rem(h, L.ce, L.rce, rem), d = max(max(L.G - q, q - (L.G + R.w - 1)), 0);
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                const int cell = in ? ((const unsigned short *)(sm + L.ol[a]))[h] : kClNone;
                const bool ok = cell != kClNone;
                c[a][u] = ok ? cell : L.ps;   // a cell whose neighbours exist
                dist[a][u] = ok ? d : 1 << 20;
                cl_row<DIM, M>(L, sm, c[a][u], w[a][u]);
                id[a][u] = ids[c[a][u]];
                b[a][u] = bs[c[a][u]];
            }
        }
    }
    __device__ __forceinline__ void first(const ClLevel<M> &L, M *x) {
#pragma unroll
        for (int u = 0; u < K; ++u)
            if (dist[0][u] <= L.D) x[c[0][u]] = b[0][u] * id[0][u];
    }
    template <int A> __device__ __forceinline__ void sweep(const ClLevel<M> &L, M *x, int d) {
#pragma unroll
        for (int u = 0; u < K; ++u)
            if (dist[A][u] <= d)
                x[c[A][u]] = cl_row_sum<DIM>(w[A][u], x, c[A][u], L.ps, L.ny, L.paired, b[A][u]) * id[A][u];
    }
    __device__ __forceinline__ void residual(const ClLevel<M> &L, const M *x, M *rs) {
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int u = 0; u < K; ++u)
                if (dist[a][u] == 0)
                    rs[c[a][u] - L.G * L.ps] = cl_residual<DIM>(w[a][u], x, c[a][u], L.ps, L.ny, L.paired, b[a][u]);
    }
    __device__ __forceinline__ void prolong(const ClLevels<M> &P, const ClLevel<M> &L, unsigned char *sm, int rank, M *x,
                                            const M *xc, int d) {
        const int q0 = cl_range(P, L, rank, L.D).q0;
#pragma unroll
        for (int u = 0; u < K; ++u)
            if (dist[0][u] <= d)
                x[c[0][u]] += xc[((const unsigned short *)(sm + L.op))[q0 * L.ce + threadIdx.x + u * blockDim.x]];
    }
};
template <int DIM, typename M> struct ClCells<DIM, M, 0> {
    const ClLevels<M> *P;
    unsigned char *sm;
    int rank;
    __device__ __forceinline__ void load(const ClLevels<M> &P_, const ClLevel<M> &, unsigned char *sm_, int rank_) {
        P = &P_;
        sm = sm_;
        rank = rank_;
    }
    template <typename F> __device__ __forceinline__ void each(const ClLevel<M> &L, int colour, int d, F f) {
        const unsigned short *lst = (const unsigned short *)(sm + L.ol[colour]);
        const ClRange R = cl_range(*P, L, rank, d);
        for (int h = R.q0 * L.ce + threadIdx.x; h < R.q1 * L.ce; h += blockDim.x) {
            const int c = lst[h];
            if (c != kClNone) f(c, h);
        }
    }
    __device__ __forceinline__ void first(const ClLevel<M> &L, M *x) {
        const M *b = (const M *)(sm + L.ob), *id = (const M *)(sm + L.oi);
        each(L, 0, L.D, [&](int c, int) { x[c] = b[c] * id[c]; });
    }
    template <int A> __device__ __forceinline__ void sweep(const ClLevel<M> &L, M *x, int d) {
        const M *b = (const M *)(sm + L.ob), *id = (const M *)(sm + L.oi);
        each(L, A, d, [&](int c, int) {
            M w[2 * DIM];
            cl_row<DIM, M>(L, sm, c, w);
            x[c] = cl_row_sum<DIM>(w, x, c, L.ps, L.ny, L.paired, b[c]) * id[c];
        });
    }
    __device__ __forceinline__ void residual(const ClLevel<M> &L, const M *x, M *rs) {
        const M *b = (const M *)(sm + L.ob);
        for (int a = 0; a < 2; ++a)
            each(L, a, 0, [&](int c, int) {
                M w[2 * DIM];
                cl_row<DIM, M>(L, sm, c, w);
                rs[c - L.G * L.ps] = cl_residual<DIM>(w, x, c, L.ps, L.ny, L.paired, b[c]);
            });
    }
    __device__ __forceinline__ void prolong(const ClLevels<M> &, const ClLevel<M> &L, unsigned char *, int, M *x, const M *xc,
                                            int d) {
        const unsigned short *par = (const unsigned short *)(sm + L.op);
        each(L, 0, d, [&](int c, int h) { x[c] += xc[par[h]]; });
    }
};

// pre-smoothing from x = 0 and the residual of the slab's cells; no barrier after it
template <int DIM, typename M, int K>
__device__ __forceinline__ void cl_pre(const ClLevels<M> &P, const ClLevel<M> &L, unsigned char *sm, int rank) {
    M *x = (M *)(sm + L.ox);
    ClCells<DIM, M, K> cells;
    cells.load(P, L, sm, rank);
    cells.first(L, x);
    __syncthreads();
    for (int s = 0; s < L.nu; ++s) {
        if (s > 0) {
            cells.template sweep<0>(L, x, L.D - 2 * s);
            __syncthreads();
        }
        cells.template sweep<1>(L, x, s == L.nu - 1 ? 1 : L.D - 2 * s - 1);   // the last one is read by the residual only
        __syncthreads();
    }
    cells.residual(L, x, (M *)(sm + P.ors));
}
// prolongation to the colour-0 cells and post-smoothing; no barrier after it
template <int DIM, typename M, int K>
__device__ __forceinline__ void cl_post(const ClLevels<M> &P, int l, unsigned char *sm, int rank) {
    const ClLevel<M> &L = P.L[l];
    M *x = (M *)(sm + L.ox);
    ClCells<DIM, M, K> cells;
    cells.load(P, L, sm, rank);
    cells.prolong(P, L, sm, rank, x, (const M *)(sm + P.L[l + 1].ox), L.E + 2 * L.nu);
    for (int s = 0; s < L.nu; ++s) {
        __syncthreads();
        cells.template sweep<1>(L, x, L.E + 2 * (L.nu - s) - 1);
        __syncthreads();
        cells.template sweep<0>(L, x, L.E + 2 * (L.nu - s) - 2);
    }
}
// entries of a colour that a thread of the CTA takes
template <typename M> __device__ __forceinline__ int cl_per_thread(const ClLevels<M> &P, const ClLevel<M> &L, int rank) {
    const ClRange R = cl_range(P, L, rank, L.D);
    return ((R.q1 - R.q0) * L.ce + (int)blockDim.x - 1) / (int)blockDim.x;
}

// b of the next level = the sum over the children's residuals (x fastest),
// stored into every CTA whose ghosts cover it (on the coarsest level, into
// every CTA's gathered copy)
template <int DIM, typename M>
__device__ __forceinline__ void cl_restrict(const ClLevels<M> &P, int l, unsigned char *sm, int rank) {
    const ClLevel<M> &L = P.L[l], &C = P.L[l + 1];
    const M *rs = (const M *)(sm + P.ors);
    const int fw = cl_range(P, L, rank, 0).w;
    const ClRange S = cl_range(P, C, rank, 0);
    const bool last = l + 1 == P.n - 1;
    M *bc = (M *)(sm + C.ob), *bx = (M *)(sm + P.obx);
    const int pl = C.ny * C.nz;
    const float rpl = 1.0f / (float)pl;
    for (int q = threadIdx.x; q < S.w * pl; q += blockDim.x) {
        int m, J;
        const int p = div_rem(q, pl, rpl, m), K = DIM == 3 ? div_rem(m, C.ny, C.rny, J) : (J = m, 0);
        const int base = p * L.rx * L.ps + J * L.ry + L.ny * (K * L.rz);
        M acc = M(0);
#pragma unroll
        for (int kk = 0; kk < (DIM == 3 ? 2 : 1); ++kk)
#pragma unroll
            for (int jj = 0; jj < 2; ++jj)
#pragma unroll
                for (int pp = 0; pp < 2; ++pp)
                    if (kk < L.rz && jj < L.ry && pp < L.rx && K * L.rz + kk < L.nz && J * L.ry + jj < L.ny &&
                        p * L.rx + pp < fw)
                        acc += rs[base + pp * L.ps + jj + L.ny * kk];
        const int i = S.s + p;
        if (last) {
            const int gc = i + C.nx * m;
            for (int r = 0; r < P.nc; ++r) cl_store(cl_addr(bx + gc, r), acc);
        } else {
            bc[(p + C.G) * C.ps + m] = acc;
            cl_push(P, C, sm, bc, i, m, C.G, rank, acc);
        }
    }
}

// x = inverse * b on the coarsest level: a warp per row, lanes over the
// columns of the inverse, two rows at a time (a CTA meets every phase once per
// iteration with few warps, so that code size costs instruction fetches:
// eight rows at a time took 3950 cycles for 5 rows per warp)
template <typename M> __device__ __forceinline__ void cl_exact(const ClLevels<M> &P, unsigned char *sm, int rank) {
    constexpr int U = 2;
    const ClLevel<M> &L = P.L[P.n - 1];
    const ClRange R = cl_range(P, L, rank, cl_exact_depth(P));
    const int ne = L.nx * L.ny * L.nz, pl = L.ny * L.nz, nr = (R.q1 - R.q0) * pl;
    const M *inv = (const M *)(sm + P.oinv), *bx = (const M *)(sm + P.obx);
    M *x = (M *)(sm + L.ox);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll 1
    for (int r0 = warp; r0 < nr; r0 += U * nw) {
        M acc[U];
#pragma unroll
        for (int u = 0; u < U; ++u) acc[u] = M(0);
        for (int m = lane; m < ne; m += 32) {
            const M v = bx[m];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (r0 + u * nw < nr) {
                    const M a = inv[(r0 + u * nw) * ne + m];
                    acc[u] = sizeof(M) == sizeof(double) ? (M)fma((double)a, (double)v, (double)acc[u]) : acc[u] + a * v;
                }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (r0 + u * nw < nr) acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], o);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int row = r0 + u * nw;
            if (lane == 0 && row < nr) {
                const int c = ((const unsigned short *)(sm + P.orow))[row];
                x[c] = acc[u];
                if (cl_exact_depth(P) < L.E) {
                    const int q = c / L.ps;
                    cl_push(P, L, sm, x, R.s - L.G + q, c - q * L.ps, L.E, rank, acc[u]);
                }
            }
        }
    }
    if (cl_exact_depth(P) < L.E) cl_sync(P.nc);
    else __syncthreads();
}

// The V-cycle over the cluster's levels. On entry the first level's b (with
// its ghosts; the gathered b when it is the coarsest) is in place and a
// cluster barrier has been passed since. On return x of the first level is
// valid on E columns beyond the slab; no barrier has been passed since its
// last half sweep.
template <int DIM, typename M>
__device__ __forceinline__ void cl_vcycle(const ClLevels<M> &P, unsigned char *sm, int rank) {
    constexpr bool F32 = sizeof(M) == sizeof(float);
    for (int l = 0; l < P.n - 1; ++l) {
        const ClLevel<M> &L = P.L[l];
        const int per = cl_per_thread(P, L, rank);
        if (per <= 1) cl_pre<DIM, M, 1>(P, L, sm, rank);
        else if (per <= 2) cl_pre<DIM, M, 2>(P, L, sm, rank);
        else if (F32 && per <= 4) cl_pre<DIM, M, F32 ? 4 : 0>(P, L, sm, rank);
        else cl_pre<DIM, M, 0>(P, L, sm, rank);
        __syncthreads();
        cl_restrict<DIM, M>(P, l, sm, rank);
        cl_sync(P.nc);
    }
    cl_exact<M>(P, sm, rank);
    for (int l = P.n - 2; l >= 0; --l) {
        const ClLevel<M> &L = P.L[l];
        const int per = cl_per_thread(P, L, rank);
        if (l < P.n - 2) __syncthreads();
        if (per <= 1) cl_post<DIM, M, 1>(P, l, sm, rank);
        else if (per <= 2) cl_post<DIM, M, 2>(P, l, sm, rank);
        else if (F32 && per <= 4) cl_post<DIM, M, F32 ? 4 : 0>(P, l, sm, rank);
        else cl_post<DIM, M, 0>(P, l, sm, rank);
    }
}

// The V-cycle below the per-level kernels: b of the first level from b_top,
// its x to x_top. The image (fixed during a solve) is copied in before the
// grid-dependency wait.
template <int DIM, typename M>
__global__ void __launch_bounds__(512, 1) k_mg_cluster(ClLevels<M> P, const M *__restrict__ b_top, M *__restrict__ x_top) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int rank = cl_rank();
    const ClLevel<M> &L = P.L[0];
    cl_load<M>(P, sm, rank);
    cp_async_wait_all();
    __syncthreads();
    griddep_wait();
    M *b = (M *)(sm + L.ob), *bx = (M *)(sm + P.obx);
    if (P.n == 1) {   // the first level is the coarsest one
        for (int c = threadIdx.x; c < L.nx * L.ny * L.nz; c += blockDim.x) bx[c] = b_top[c];
    } else {
        const int s = cl_start(P, L, rank);
        for (int c = threadIdx.x; c < L.ncol * L.ny * L.nz; c += blockDim.x) {
            int q, j, k;
            split3(c, L.ncol, L.rncol, L.ny, L.rny, q, j, k);
            const int i = s - L.G + q;
            if (i >= 0 && i < L.nx) b[q * L.ps + j + L.ny * k] = b_top[i + L.nx * (j + L.ny * k)];
        }
    }
    cl_sync(P.nc);   // and every CTA's shared memory is ready for remote stores
    cl_vcycle<DIM, M>(P, sm, rank);
    __syncthreads();
    const ClRange R = cl_range(P, L, rank, 0);
    const M *x = (const M *)(sm + L.ox);
    const float rw = 1.0f / (float)R.w;
    for (int c = threadIdx.x; c < R.w * L.ny * L.nz; c += blockDim.x) {
        int q, j, k;
        split3(c, R.w, rw, L.ny, L.rny, q, j, k);
        x_top[R.s + q + L.nx * (j + L.ny * k)] = x[(q + L.G) * L.ps + j + L.ny * k];
    }
}

// ---------------------------------------------------------------------------
// a whole pressure solve of a small 2D grid in one cluster
// ---------------------------------------------------------------------------
// On such grids a PCG iteration is 11 to 20 dependent launches of 1.2 to 10 us,
// and the solve's loops are conditional graph nodes (about 5 us to enter and to
// leave one). Here level 0 joins the cluster's levels and the vectors of the
// PCG live in shared memory as well; an iteration has one cluster barrier per
// level and one per dot product. The arithmetic is that of k_cg_init,
// k_cg_pz_apply (mixed) or k_cg_pupdate and k_cg_apply_dot (FP64), k_cg_update
// and k_cg_refine. On the mixed path the dot products also sum the same groups
// of cells in FP32 as a thread of those kernels does, and the groups in
// compensated pairs, so alpha and beta round to the same FP32 values: FP32
// rounding inside the V-cycle is amplified in the smoothest pressure mode, and
// only the same operands give the same pressure.
struct ClSolve {
    GridD g;
    const uint32_t *info;
    C3<double> w64;
    double *q;            // pressure, in and out
    const double *b;
    double *r64;          // mixed path: FP64 residual
    double *scal;
    int *ctl;
    double rtol, inv_nf;  // inv_nf > 0: also E_k (k_cg_init)
    int maxit, by;        // by: rows per block of the launched CG kernels (their threads' groups of cells)
    int op, oap, oe;      // shared memory: p, Ap, e (mixed): the slab and one column on each side
};
struct ClControl {        // one per CTA, written by its thread 0 from totals all CTAs share
    double target, itarget, rz0, rz1;
    double test2;         // square of the norm the iteration stops at
    double rrz;           // 1 / rz1
    double alpha, beta;
    float alpha_f, beta_f;
    int more;
};

// totals over the cluster of nv FP64 values per thread (at most four; a warp
// sums each), valid in warp 0 of every CTA (same order everywhere: same
// result). Two buffers, alternating: a CTA may store for the next reduction
// while another still reads this one. aside() is called by a warp that does
// not sum.
struct ClNothing { __device__ __forceinline__ void operator()() const {} };
template <typename M, typename F = ClNothing>
__device__ __forceinline__ void cl_sum(const ClLevels<M> &P, unsigned char *sm, int rank, int &buf, double *v, int nv,
                                       F aside = F()) {
    const int t = threadIdx.x, nt = blockDim.x, warp = t >> 5, lane = t & 31;
    double *sh = (double *)(sm + P.ored), *slot = sh + 4 * nt + buf * 4 * kMaxCluster;
    for (int q = 0; q < nv; ++q) sh[q * nt + t] = v[q];
    __syncthreads();
    if (warp < nv) {
        const double *a = sh + warp * nt;
        double s = 0.0;   // blocks of 128 k threads
        for (int m = lane; m < nt; m += 128) s += (a[m] + a[m + 32]) + (a[m + 64] + a[m + 96]);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane < P.nc) cl_store(cl_addr(slot + warp * kMaxCluster + rank, lane), s);
    } else if (warp == 4) aside();
    cl_sync(P.nc);
    if (warp == 0)
        for (int q = 0; q < nv; ++q) {
            double s = lane < P.nc ? slot[q * kMaxCluster + lane] : 0.0;
            for (int o = P.nc >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            v[q] = s;
        }
    buf ^= 1;
}
// the same for one value of the vectors' type: FP64 as above, FP32 in
// compensated pairs; the total is valid in thread 0
template <typename M, typename F = ClNothing>
__device__ __forceinline__ double cl_dot(const ClLevels<M> &P, unsigned char *sm, int rank, int &buf, DotAcc64 a, F aside = F()) {
    cl_sum(P, sm, rank, buf, &a.s, 1, aside);
    return a.s;
}
template <typename M, typename F = ClNothing>
__device__ __forceinline__ double cl_dot(const ClLevels<M> &P, unsigned char *sm, int rank, int &buf, DotAcc32 a, F aside = F()) {
    const int t = threadIdx.x, nw = blockDim.x >> 5, warp = t >> 5, lane = t & 31;
    float2 *sh = (float2 *)(sm + P.ored), *slot = (float2 *)((double *)(sm + P.ored) + 4 * blockDim.x + buf * 4 * kMaxCluster);
    auto tree = [](float &s, float &e, int from) {
#pragma unroll 1
        for (int o = from; o > 0; o >>= 1) {
            const float so = __shfl_xor_sync(0xffffffffu, s, o), eo = __shfl_xor_sync(0xffffffffu, e, o);
            float sn, se;
            two_sum(s, so, sn, se);
            s = sn;
            e += eo + se;
        }
    };
    float s = a.s, e = a.e;
    tree(s, e, 16);
    if (lane == 0) sh[warp] = make_float2(s, e);
    __syncthreads();
    if (warp == 0) {
        s = lane < nw ? sh[lane].x : 0.f;
        e = lane < nw ? sh[lane].y : 0.f;
        tree(s, e, 16);
        if (lane < P.nc) {
            const unsigned d = cl_addr(slot + rank, lane);
            cl_store(d, s);
            cl_store(d + 4, e);
        }
    } else if (warp == 4) aside();
    cl_sync(P.nc);
    double tot = 0.0;
    if (warp == 0) {
        s = lane < P.nc ? slot[lane].x : 0.f;
        e = lane < P.nc ? slot[lane].y : 0.f;
        tree(s, e, P.nc >> 1);
        if (t == 0) tot = (double)s + (double)e;
    }
    buf ^= 1;
    return tot;
}

// own cells of level 0: own column pc, row j, x fastest (rows of the global arrays)
#define CL_OWN_CELLS()                                                                                        \
    for (int g_ = t, pc, j, k_; g_ < S.w * L.ny && (split3(g_, S.w, rw, L.ny, L.rny, pc, j, k_), true); g_ += blockDim.x)

// own cells of level 0, a column after the other: position o = pc ps + j in the
// slab's columns, local cell o + G ps
#define CL_COLUMN_CELLS()                                                                                     \
    for (int g_ = t, pc, j, o; g_ < S.w * L.ny && (pc = div_rem(g_, L.ny, L.rny, j), o = pc * ps + j, true); g_ += blockDim.x)

// sums of the groups of own cells that one thread of the launched CG kernels
// takes (launch_groups): products f of own column pc, rows j0 + u by for u < rpt
template <typename T>
__device__ __forceinline__ typename DotAcc<T>::type cl_group_sums(const T *f, int w, int ny, int ps, int by, int rpt) {
    typename DotAcc<T>::type acc;
    const int nb = (ny + by * rpt - 1) / (by * rpt), ng = by * nb;
    const float rng = 1.0f / (float)ng, rby = 1.0f / (float)by;
    for (int g = threadIdx.x; g < w * ng; g += blockDim.x) {
        int m, ty;
        const int pc = div_rem(g, ng, rng, m), blk = div_rem(m, by, rby, ty);
        T a = T(0);
        for (int u = 0, j = blk * by * rpt + ty; u < rpt && j < ny; ++u, j += by) a += f[pc * ps + j];
        acc.add(a);
    }
    return acc;
}

template <typename T>
__global__ void __launch_bounds__(512, 1) k_solve_cluster(ClLevels<T> P, ClSolve A) {
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ ClControl K;
    constexpr bool MIXED = sizeof(T) == sizeof(float);
    const int rank = cl_rank(), t = threadIdx.x;
    const ClLevel<T> &L = P.L[0];
    const int ps = L.ps;
    const ClRange S = cl_range(P, L, rank, 0);
    cl_load<T>(P, sm, rank);
    T *x = (T *)(sm + L.ox), *r = (T *)(sm + L.ob), *bx = (T *)(sm + P.obx);
    T *p = (T *)(sm + A.op) - (L.G - 1) * ps, *Ap = (T *)(sm + A.oap) - (L.G - 1) * ps, *e = (T *)(sm + A.oe) - (L.G - 1) * ps;
    for (int c = t + (L.G - 1) * ps; c < (L.G + S.w + 1) * ps; c += blockDim.x) { p[c] = T(0); Ap[c] = T(0); }
    T *prod = (T *)(sm + P.ors);   // products of a dot, by own cell
    const float rw = 1.0f / (float)S.w;
    int buf = 0, its = 0, outer = 0, nan_seen = 0, notconv = 0;
    cp_async_wait_all();
    cl_sync(P.nc);   // every CTA's shared memory is ready for remote stores
    griddep_wait();

    // residual of an own cell, with the copies the ghosts (or, when level 0 is
    // the coarsest, the gathered right-hand side) need
    auto put_r = [&](int pc, int j, T rc) {
        r[(pc + L.G) * ps + j] = rc;
        if (P.n == 1)
            for (int m = 0; m < P.nc; ++m) cl_store(cl_addr(bx + S.s + pc + L.nx * j, m), rc);
        else
            cl_push(P, L, sm, r, S.s + pc, j, L.G, rank, rc);
    };

    double qbar = 0.0, qsum[1] = {0.0};
    if (A.inv_nf > 0.0) {
        CL_OWN_CELLS() qsum[0] += A.q[S.s + pc + L.nx * j];
        cl_sum(P, sm, rank, buf, qsum, 1);
        if (t == 0) K.rz0 = qsum[0];
        __syncthreads();
        qbar = K.rz0 * A.inv_nf;
    }
    double acc[4] = {0.0, 0.0, 0.0, 0.0};   // b.b, r.r, sum |b - Mq|, the normalisation
    CL_OWN_CELLS() {
        const int i = S.s + pc, gc = i + L.nx * j;
        const uint32_t inf = A.info[gc];
        double rc = 0.0;
        if (inf & INFO_FLUID) {
            const double bc = A.b[gc];
            const double Mq = poisson_row64<2>(A.g, inf, gc, i, j, 0, A.w64, A.q);
            rc = bc - Mq;
            acc[0] = fma(bc, bc, acc[0]);
            acc[1] = fma(rc, rc, acc[1]);
            if (A.inv_nf > 0.0) {
                const double Mqbar = ftype(inf, 0, 1) == FT_OUTLET ? qbar * A.w64.a[0][fhi(A.g, 0, i, j, 0)] : 0.0;
                acc[2] += fabs(bc - Mq);
                acc[3] += fabs(Mq - Mqbar) + fabs(bc - Mqbar);
            }
        }
        if (MIXED) A.r64[gc] = rc;
        put_r(pc, j, (T)rc);
    }
    cl_sum(P, sm, rank, buf, acc, A.inv_nf > 0.0 ? 4 : 2);
    if (t == 0) {
        const double bn = sqrt(acc[0]), rn = sqrt(acc[1]);
        const bool bad = !(isfinite(bn) && isfinite(rn));
        K.target = A.rtol * (bn > 0.0 ? bn : rn);
        K.itarget = fmax(kInnerRtol * rn, kTripMargin * K.target);
        K.test2 = MIXED ? K.itarget * K.itarget : K.target * K.target;
        K.rz0 = 0.0;
        K.more = !bad && rn > K.target;
        nan_seen |= bad;
        if (rank == 0) {
            A.scal[S_BB] = acc[0];
            A.scal[S_RR] = acc[1];
            A.scal[S_TARGET] = K.target;
            if (A.inv_nf > 0.0) {
                A.scal[S_QSUM] = qsum[0];
                A.scal[S_RES] = acc[2];
                A.scal[S_NRM] = acc[3];
                A.scal[S_E] = acc[2] / (acc[3] + 1e-20);
            }
        }
    }
    __syncthreads();
    while (K.more) {   // mixed: defect-correction trips; FP64: one pass
        int it = 0;
        do {
            cl_vcycle<2, T>(P, sm, rank);
            __syncthreads();
            typename DotAcc<T>::type dz;   // r.z: a colour-0 cell with its row partner (level 0 on its own: cell by cell)
            for (int g = t; g < ((S.w + 1) >> 1) * L.ny; g += blockDim.x) {
                int j;
                const int tp = div_rem(g, L.ny, L.rny, j), lo = (2 * tp + L.G) * ps + j, odd = (S.s + j) & 1;
                const bool two = 2 * tp + 1 < S.w;
                const int ca = odd ? lo + ps : lo, cb = odd ? lo : lo + ps;   // colour 0, colour 1
                T a = T(0);
                if (!odd || two) a = r[ca] * x[ca];
                if (L.paired) { dz.add(a); a = T(0); }
                if (odd || two) a += r[cb] * x[cb];
                dz.add(a);
            }
            const double rz = cl_dot(P, sm, rank, buf, dz);
            if (t == 0) {
                K.rz1 = rz;
                K.beta = K.rz0 != 0.0 ? rz * K.rrz : 0.0;
                K.beta_f = (float)K.beta;
            }
            __syncthreads();
            typename DotAcc<T>::type dp;
            const T *c0 = (const T *)(sm + L.oc[0]), *c1 = (const T *)(sm + L.oc[1]);
            if constexpr (MIXED) {   // p = z + beta p, Ap = M z + beta Ap, p.Ap
                const T be = K.beta_f;
                const bool fresh = be == T(0);
                CL_COLUMN_CELLS() {
                    const int c = o + L.G * ps;
                    const T zc = x[c];
                    const T pn = fresh ? zc : zc + be * p[c];
                    T y = c0[c] * (zc - x[c - ps]);
                    y += c0[c + ps] * (zc - x[c + ps]);
                    y += c1[c] * (zc - x[c - 1]);
                    y += c1[c + 1] * (zc - x[c + 1]);
                    const T an = fresh ? y : y + be * Ap[c];
                    p[c] = pn;
                    Ap[c] = an;
                    prod[o] = pn * an;
                }
                __syncthreads();
                dp = cl_group_sums<T>(prod, S.w, L.ny, ps, A.by, kApplyRows);
            } else {   // p = z + beta p (one ghost column as well), Ap = M p, p.Ap
                const T be = K.beta;
                for (int c = t + (L.G - 1) * ps; c < (L.G + S.w + 1) * ps; c += blockDim.x) p[c] = x[c] + be * p[c];
                __syncthreads();
                CL_COLUMN_CELLS() {
                    const int c = o + L.G * ps;
                    const T pv = p[c];
                    T y = c0[c] * (pv - p[c - ps]);
                    y += c0[c + ps] * (pv - p[c + ps]);
                    y += c1[c] * (pv - p[c - 1]);
                    y += c1[c + 1] * (pv - p[c + 1]);
                    Ap[c] = y;
                    dp.add(pv * y);
                }
            }
            const double pap = cl_dot(P, sm, rank, buf, dp);
            if (t == 0) {
                K.alpha = K.rz1 / pap;
                K.alpha_f = (float)K.alpha;
            }
            __syncthreads();
            const T al = MIXED ? (T)K.alpha_f : (T)K.alpha;
            typename DotAcc<T>::type dr;
            CL_COLUMN_CELLS() {   // x += alpha p, r -= alpha Ap, r.r
                const int c = o + L.G * ps;
                if constexpr (MIXED) e[c] = it == 0 ? al * p[c] : e[c] + al * p[c];
                else A.q[S.s + pc + L.nx * j] += al * p[c];
                const T rc = r[c] - al * Ap[c];
                put_r(pc, j, rc);
                if constexpr (MIXED) prod[o] = rc * rc;
                else dr.add(rc * rc);
            }
            if constexpr (MIXED) {
                __syncthreads();
                dr = cl_group_sums<T>(prod, S.w, L.ny, ps, A.by, kUpdateRows);
            }
            const double rr = cl_dot(P, sm, rank, buf, dr, [&] { if (t == 128) K.rrz = 1.0 / K.rz1; });
            ++it;
            ++its;
            if (t == 0) {
                K.rz0 = K.rz1;
                const bool bad = !isfinite(rr);
                nan_seen |= bad;
                bool more = !bad && rr > K.test2;
                if (more && it >= A.maxit) { notconv = 1; more = false; }
                K.more = more;
                if (rank == 0) A.scal[S_RR] = rr;
            }
            __syncthreads();
        } while (K.more);
        if constexpr (!MIXED) break;
        else {
            // end of a trip: q += e, r64 -= M e (compensated), the FP64 test
            CL_OWN_CELLS() {
                const int c = (pc + L.G) * ps + j;
                x[c] = e[c];
                cl_push(P, L, sm, x, S.s + pc, j, 1, rank, e[c]);
            }
            cl_sync(P.nc);
            const T *c0 = (const T *)(sm + L.oc[0]), *c1 = (const T *)(sm + L.oc[1]);
            double rr[1] = {0.0};
            CL_OWN_CELLS() {
                const int c = (pc + L.G) * ps + j, gc = S.s + pc + L.nx * j;
                const float ec = e[c];
                const float w[4] = {c0[c], c0[c + ps], c1[c], c1[c + 1]};
                const float en[4] = {x[c - ps], x[c + ps], x[c - 1], x[c + 1]};
                float s = 0.f, cc = 0.f;
#pragma unroll
                for (int f = 0; f < 4; ++f) {   // the faces and order of poisson_row_comp
                    float dh, lo, pp, pe, sn, se;
                    two_sum(ec, -en[f], dh, lo);
                    two_prod(w[f], dh, pp, pe);
                    pe += w[f] * lo;
                    two_sum(s, pp, sn, se);
                    s = sn;
                    cc += se + pe;
                }
                A.q[gc] += (double)ec;
                const double rn = A.r64[gc] - ((double)s + (double)cc);
                A.r64[gc] = rn;
                r[c] = (float)rn;
                rr[0] = fma(rn, rn, rr[0]);
            }
            cl_sum(P, sm, rank, buf, rr, 1);
            ++outer;
            if (t == 0) {
                const double rn = sqrt(rr[0]);
                const bool bad = !isfinite(rn);
                nan_seen |= bad;
                bool more = !bad && rn > K.target;
                if (more && outer >= kMaxOuter) { notconv = 1; more = false; }
                K.itarget = fmax(kInnerRtol * rn, kTripMargin * K.target);
                K.test2 = K.itarget * K.itarget;
                K.rz0 = 0.0;
                K.more = more;
                if (rank == 0) A.scal[S_RR] = rr[0];
            }
            CL_OWN_CELLS() put_r(pc, j, r[(pc + L.G) * ps + j]);
            cl_sync(P.nc);
        }
    }
    if (rank == 0 && t == 0) {
        A.ctl[C_IT] = its;
        A.ctl[C_ITSUM] += its;
        A.ctl[C_OUT] = outer;
        A.ctl[C_OSUM] += outer;
        if (nan_seen) A.ctl[C_NAN] = 1;
        if (notconv) A.ctl[C_NOTCONV] = 1;
    }
    cl_sync(P.nc);   // no CTA leaves while a neighbour may still store into its shared memory
}

// ---------------------------------------------------------------------------
// the coarsest level's explicit inverse
// ---------------------------------------------------------------------------
// Formed on the first PISO set-up of a step call and every refresh-th one
// after it (ctl[C_PACK], advanced by k_cl_pack, counts them); in between the
// stored inverse is kept (a preconditioner component: a stale one changes
// iterations, not the solution).

// f(0), ..., f(N - 1) with the index a constant from the start, so that an
// array it indexes is a set of registers (choices between elements of a loop
// unrolled later are made by address, which puts the array in local memory)
template <int I> struct Idx {
    __host__ __device__ constexpr operator int() const { return I; }
};
template <typename F, int... I> __device__ __forceinline__ void static_for(F f, std::integer_sequence<int, I...>) {
    (f(Idx<I>{}), ...);
}
template <int N, typename F> __device__ __forceinline__ void static_for(F f) {
    static_for(f, std::make_integer_sequence<int, N>{});
}

// FP32: Gauss-Jordan elimination without pivoting, in place (the matrix is
// symmetric positive definite: the fluid is connected to the Dirichlet
// outlet). Rows of cells that are solid or have no coefficients decouple; a
// pivot that vanishes (a pocket cut off from the outlet) drops its row and
// column. One CTA; each thread keeps an 8x8 tile of the matrix in registers,
// and the pivots go eight at a time: the 8x8 pivot tile (one warp), then its
// rows and columns (a thread per column and per row), then the eight rank-one
// updates of every other tile, four block barriers per eight pivots: 84 us at
// 128 cells. (Pivot by pivot, one barrier each: 143 us; with the matrix in
// shared memory: 240 us.) Every entry sees
// the same operations in the same order whatever the grouping.
constexpr int kGjThreads = 256, kGjTile = 8;
template <int DIM>
__global__ void __launch_bounds__(kGjThreads) k_mg_inverse_dense(GridD g, MG3<float> cc, const float *__restrict__ diag,
                                                                 const uint8_t *__restrict__ fluid,
                                                                 float *__restrict__ inv, int refresh,
                                                                 const int *__restrict__ ctl) {
    static_assert(kGjThreads * kGjTile * kGjTile == kExactCells * kExactCells, "tiles cover the matrix");
    constexpr int B = kGjTile, TC = kExactCells / B;
    griddep_wait();
    if (ctl[C_PACK] % refresh != 0) return;
    // panels of the pivot tile's rows and columns; per pivot: the multipliers
    // of every row and the normalised pivot row
    __shared__ __align__(16) float ak[B][kExactCells], nk[B][kExactCells], rowp[B][kExactCells];
    __shared__ float colp[kExactCells][B + 1];
    __shared__ float pa[B][B], pn[B][B], pinv_s[B];   // the same inside the pivot tile, and the reciprocal pivots
    const int t = threadIdx.x, n = g.ncell, ti = t / TC, tj = t % TC, i0 = ti * B, j0 = tj * B;
    // the (at most 2 DIM + 1) entries of every row, one thread per row
    __shared__ int ecol[kExactCells][2 * DIM + 1];
    __shared__ float eval[kExactCells][2 * DIM + 1];
    for (int r = t; r < kExactCells; r += kGjThreads) {
        const int i = r % g.nx, j = (r / g.nx) % g.ny, k = r / (g.nx * g.ny);
        const int ijk[3] = {i, j, k}, e[3] = {g.nx, g.ny, g.nz};
        const float d = r < n ? diag[r] : 0.f;
        const bool live = r < n && fluid[r] && d > 0.f;
        ecol[r][2 * DIM] = live ? r : -1;
        eval[r][2 * DIM] = d;
#pragma unroll
        for (int q = 0; q < DIM; ++q) {
            const int off = noff(g, q);
            const float wl = live && ijk[q] > 0 ? cc.a[q][flo(g, q, i, j, k)] : 0.f;
            const float wh = live && ijk[q] < e[q] - 1 ? cc.a[q][fhi(g, q, i, j, k)] : 0.f;
            ecol[r][2 * q] = wl != 0.f ? r - off : -1;   // a zero coefficient (wall) is no entry
            ecol[r][2 * q + 1] = wh != 0.f ? r + off : -1;
            eval[r][2 * q] = -wl;
            eval[r][2 * q + 1] = -wh;
        }
    }
    __syncthreads();
    float A[B * B];
    static_for<B>([&](auto u) {
        static_for<B>([&](auto v) { A[u * B + v] = 0.f; });
        static_for<2 * DIM + 1>([&](auto m) {
            const int c = ecol[i0 + u][m] - j0;
            const float w = eval[i0 + u][m];
            static_for<B>([&](auto v) { A[u * B + v] = c == v ? w : A[u * B + v]; });
        });
    });
#pragma unroll 1
    for (int kb = 0; kb * B < n; ++kb) {
        if (ti == kb) static_for<B * B>([&](auto q) { rowp[q / B][j0 + q % B] = A[q]; });
        if (tj == kb) static_for<B * B>([&](auto q) { colp[i0 + q / B][q % B] = A[q]; });
        __syncthreads();
        if (t < 32) {   // the pivot tile: lane v < 8 holds its column v
            const int v = t & (B - 1);
            float p[B];
            static_for<B>([&](auto u) { p[u] = rowp[u][kb * B + v]; });
            static_for<B>([&](auto k) {
                const float pv = __shfl_sync(0xffffffffu, p[k], k);
                const float pinv = pv > 0.f ? 1.f / pv : 0.f;   // a vanished pivot zeroes its row and column
                const float nv = p[k] * pinv;
                static_for<B>([&](auto u) {
                    const float a = __shfl_sync(0xffffffffu, p[u], k);
                    if (t == 0) pa[k][u] = a;
                    p[u] = v == k ? -a * pinv : fmaf(-a, nv, p[u]);
                });
                p[k] = v == k ? pinv : nv;
                if (t < B) pn[k][v] = nv;
                if (t == 0) pinv_s[k] = pinv;
            });
            if (t < B) static_for<B>([&](auto u) { rowp[u][kb * B + v] = p[u]; });
        }
        __syncthreads();
        if (t < kExactCells) {   // column t of the pivot rows
            const int j = t;
            if (j / B == kb) {
                static_for<B>([&](auto k) { nk[k][j] = pn[k][j - kb * B]; });
            } else {
                float r[B];
                static_for<B>([&](auto u) { r[u] = rowp[u][j]; });
                static_for<B>([&](auto k) {
                    const float v = r[k] * pinv_s[k];
                    nk[k][j] = v;
                    static_for<B>([&](auto u) { r[u] = u == k ? v : fmaf(-pa[k][u], v, r[u]); });
                });
                static_for<B>([&](auto u) { rowp[u][j] = r[u]; });
            }
        } else {                 // row i of the pivot columns
            const int i = t - kExactCells;
            if (i / B != kb) {
                float c[B];
                static_for<B>([&](auto v) { c[v] = colp[i][v]; });
                static_for<B>([&](auto k) {
                    const float a = c[k];
                    ak[k][i] = a;
                    static_for<B>([&](auto v) { c[v] = v == k ? -a * pinv_s[k] : fmaf(-a, pn[k][v], c[v]); });
                });
                static_for<B>([&](auto v) { colp[i][v] = c[v]; });
            }
        }
        __syncthreads();
        if (ti == kb) {
            static_for<B * B>([&](auto q) { A[q] = rowp[q / B][j0 + q % B]; });
        } else if (tj == kb) {
            static_for<B * B>([&](auto q) { A[q] = colp[i0 + q / B][q % B]; });
        } else {
#pragma unroll 2
            for (int k = 0; k < B; ++k) {
                const float4 a0 = *(const float4 *)&ak[k][i0], a1 = *(const float4 *)&ak[k][i0 + 4];
                const float4 v0 = *(const float4 *)&nk[k][j0], v1 = *(const float4 *)&nk[k][j0 + 4];
                const float a[B] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
                const float v[B] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
                static_for<B * B>([&](auto q) { A[q] = fmaf(-a[q / B], v[q % B], A[q]); });
            }
        }
        __syncthreads();
    }
    static_for<B * B>([&](auto q) {
        if (i0 + q / B < n && j0 + q % B < n) inv[(i0 + q / B) * n + j0 + q % B] = A[q];
    });
}

// FP64: LDL^T without pivoting in band form, cells ordered with the shortest
// axis fastest, so that the band is the product of the two shortest extents (4
// to 25 for at most 128 cells), then L D L^T x = e_j for every column j of the
// inverse: n^2 (2 bw + 1) operations instead of the n^3 of a dense elimination,
// which the SM's two FP64 FMAs per clock take 1.1 ms for at 128 cells. What is
// left is a serial chain along the cells, halved by working from both ends: h
// cells from the first and h from the last one on, by the two halves of a warp
// in the same instructions, then the bw or bw + 1 cells between them. A column
// of the factor costs a division and two FMAs in a row, a cell of a solve one
// FMA (a thread keeps the last bw values of its column in registers, the
// newest one's term added last; the next cell's factors are loaded before).
// A block is one warp with 16 columns of the inverse, the factorisation
// repeated in each: several warps on one SM would be bound by its FP64 rate.
// 60 us for 32x4 cells, 98 for 16x8, 333 for 5x5x5 (from one end alone 130, 182
// and 643 us).
// Rows of cells that are solid or have no coefficients, and of pivots that
// vanish (against the diagonal they came from), give a zero row and column.
constexpr int kBandCols = 16;
// the rows of the factor a half keeps, and the shared memory of the kernel
struct BandShape { int n, bw, h, s, rows; };   // s cells in the middle; rows = h + s of either half
__host__ __device__ inline BandShape band_shape(int n, int bw) {
    BandShape b;
    b.n = n;
    b.bw = bw;
    b.h = n > bw ? (n - bw) / 2 : 0;
    b.s = n - 2 * b.h;
    b.rows = b.h + b.s;
    return b;
}
// per half: the matrix rows (bw + 1 each) and the factor (bw each) and pivots;
// the columns of the inverse
__host__ __device__ inline size_t band_words(const BandShape &b) {
    return 2 * (size_t)b.rows * (2 * b.bw + 3) + (size_t)b.n * kBandCols;
}
// Substitution over count rows: row q takes start(q) less the products of
// load(q, d) with the value d rows back (win[d - 1]), and goes to store(q). The
// operands of a row are loaded while the row before is worked.
template <typename M, int W, typename FL, typename FA, typename FS>
__device__ __forceinline__ void band_rows(M (&win)[W], int bw, int count, FL load, FA start, FS store) {
    M l[W], ln[W];
#pragma unroll
    for (int d = 0; d < W; ++d) l[d] = M(0);
    if (count > 0) {
#pragma unroll
        for (int d = 0; d < W; ++d) if (d < bw) l[d] = load(0, d + 1);
    }
    M a = count > 0 ? start(0) : M(0);
#pragma unroll 1
    for (int q = 0; q < count; ++q) {
        M an = M(0);
#pragma unroll
        for (int d = 0; d < W; ++d) ln[d] = M(0);
        if (q + 1 < count) {
#pragma unroll
            for (int d = 0; d < W; ++d) if (d < bw) ln[d] = load(q + 1, d + 1);
            an = start(q + 1);
        }
#pragma unroll
        for (int d = W; d >= 1; --d) a = fma(-l[d - 1], win[d - 1], a);   // entries beyond the band are 0
        store(q, a);
#pragma unroll
        for (int d = W - 1; d > 0; --d) win[d] = win[d - 1];
        win[0] = a;
#pragma unroll
        for (int d = 0; d < W; ++d) l[d] = ln[d];
        a = an;
    }
}
// one column of the inverse per thread pair (t, t + 16): half 0 works the rows
// from the first cell on, half 1 those from the last one on (its row q is band
// row n - 1 - q), both the middle rows
template <typename M, int W>
__device__ __forceinline__ void band_solve(const BandShape S, const M *L0, const M *L1, const M *D0, const M *D1, M *Y, int col, bool live) {
    const int t = threadIdx.x, half = t / kBandCols, lane = t % kBandCols, bw = S.bw, h = S.h, s = S.s, n = S.n;
    const M *L = half ? L1 : L0, *D = half ? D1 : D0;   // L[i bw + d - 1] = L(i, i - d)
    const int mine = half ? n - 1 - col : col;          // the unit entry, in this half's row order
    auto y = [&](int q) -> M & { return Y[(half ? n - 1 - q : q) * kBandCols + lane]; };
    M win[W];
#pragma unroll
    for (int d = 0; d < W; ++d) win[d] = M(0);
    // forward over this half's rows
    band_rows<M, W>(win, bw, h, [&](int q, int d) { return L[q * bw + d - 1]; },
                          [&](int q) { return live && q == mine ? M(1) : M(0); }, [&](int q, M a) { y(q) = a; });
    // what they put into the middle rows: half 0 leaves it in Y, half 1 adds
    M mid[W + 1];
#pragma unroll
    for (int q = 0; q <= W; ++q) {
        M a = M(0);
        if (q < s) {
#pragma unroll
            for (int d = W; d >= 1; --d)
                if (d <= bw && d > q) a = fma(-L[(h + q) * bw + d - 1], win[d > q ? d - 1 - q : 0], a);
        }
        mid[q] = a;
    }
    if (half == 0) {
#pragma unroll
        for (int q = 0; q <= W; ++q)
            if (q < s) Y[(h + q) * kBandCols + lane] = mid[q] + (live && h + q == col ? M(1) : M(0));
    }
    __syncwarp();
    if (half == 1) {
#pragma unroll
        for (int q = 0; q <= W; ++q)
            if (q < s) Y[(h + s - 1 - q) * kBandCols + lane] += mid[q];
    }
    __syncwarp();
    if (half == 0) {   // the middle rows: forward, then back
#pragma unroll
        for (int d = 0; d < W; ++d) win[d] = M(0);
        band_rows<M, W>(win, bw, s, [&](int q, int d) { return q >= d ? L0[(h + q) * bw + d - 1] : M(0); },
                              [&](int q) { return Y[(h + q) * kBandCols + lane]; },
                              [&](int q, M a) { Y[(h + q) * kBandCols + lane] = a; });
#pragma unroll
        for (int d = 0; d < W; ++d) win[d] = M(0);
        band_rows<M, W>(win, bw, s,
                              [&](int q, int d) { return q >= d ? L0[(h + s - 1 - q + d) * bw + d - 1] : M(0); },
                              [&](int q) { return Y[(h + s - 1 - q) * kBandCols + lane] * D0[h + s - 1 - q]; },
                              [&](int q, M a) { Y[(h + s - 1 - q) * kBandCols + lane] = a; });
    }
    __syncwarp();
    // back over this half's rows
#pragma unroll
    for (int d = 0; d < W; ++d) win[d] = d < s && d < bw ? y(h + d) : M(0);
    band_rows<M, W>(win, bw, h, [&](int q, int d) { return L[(h - 1 - q + d) * bw + d - 1]; },
                          [&](int q) { return y(h - 1 - q) * D[h - 1 - q]; }, [&](int q, M a) { y(h - 1 - q) = a; });
    __syncwarp();
}
template <int DIM, typename M>
__global__ void __launch_bounds__(32) k_mg_inverse_band(GridD g, MG3<M> cc, const M *__restrict__ diag,
                                                        const uint8_t *__restrict__ fluid, M *__restrict__ inv, int refresh,
                                                        const int *__restrict__ ctl) {
    extern __shared__ __align__(16) unsigned char sm[];
    griddep_wait();
    if (ctl[C_PACK] % refresh != 0) return;
    const int t = threadIdx.x, n = g.ncell;
    // axes by extent, shortest first
    int ax[3] = {0, 1, 2};
    const int e[3] = {g.nx, g.ny, g.nz};
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int q = 0; q < 2; ++q)
            if (e[ax[q]] > e[ax[q + 1]]) { const int s = ax[q]; ax[q] = ax[q + 1]; ax[q + 1] = s; }
    int st[3];   // stride of axis a in the band order
    st[ax[0]] = 1;
    st[ax[1]] = e[ax[0]];
    st[ax[2]] = e[ax[0]] * e[ax[1]];
    const int bw = st[ax[2]], W = bw + 1;
    const BandShape S = band_shape(n, bw);
    // rows of a half: A[i W + d] = A(i, i - d), then the Schur complement;
    // L[i bw + d - 1] = L(i, i - d); rD = reciprocal pivots. Half 1 counts rows
    // and columns from the last cell back
    const int half = t / kBandCols, lane = t % kBandCols;
    M *A0 = (M *)sm, *A1 = A0 + S.rows * W, *L0 = A1 + S.rows * W, *L1 = L0 + S.rows * bw, *D0 = L1 + S.rows * bw;
    M *D1 = D0 + S.rows, *T0 = D1 + S.rows, *T1 = T0 + S.rows, *Y = T1 + S.rows;   // T: pivots below it vanish
    __shared__ int cell_s[kExactCells];   // cell of a band index
    __shared__ unsigned short tri_s[kExactCells * 4];   // (u, v), v <= u, of the entries of a column's update
    const int total = 2 * S.rows * (2 * bw + 3);
    for (int q = t; q < total; q += 32) A0[q] = M(0);
    for (int u = t; u < bw; u += 32)
        for (int v = 0; v <= u; ++v) tri_s[u * (u + 1) / 2 + v] = (unsigned short)(u << 8 | v);
    __syncwarp();
    for (int c = t; c < n; c += 32) {
        const int i = c % g.nx, j = (c / g.nx) % g.ny, k = c / (g.nx * g.ny);
        const int r = i * st[0] + j * st[1] + k * st[2], rr = n - 1 - r;
        cell_s[r] = c;
        const M d = diag[c];
        const bool live = fluid[c] && d > M(0);
        if (!live) continue;
        const M tiny = d * M(1e-13);
        if (r < S.rows) {
            A0[r * W] = d;
            T0[r] = tiny;
        } else {
            A1[rr * W] = d;
            T1[rr] = tiny;
        }
        const int ijk[3] = {i, j, k};
#pragma unroll
        for (int a = 0; a < DIM; ++a) {   // the low neighbour is the one of smaller band index
            if (ijk[a] == 0) continue;
            const M w = -cc.a[a][flo(g, a, i, j, k)];
            if (r < S.rows) A0[r * W + st[a]] = w;
            else A1[(n - 1 - (r - st[a])) * W + st[a]] = w;   // row r - st[a] of half 1: st[a] after r
        }
    }
    __syncwarp();
    // right-looking: after step k the columns beyond k hold the Schur
    // complement and column k of L the factor
    const int np = bw * (bw + 1) / 2;
    M *A = half ? A1 : A0, *L = half ? L1 : L0, *D = half ? D1 : D0, *T = half ? T1 : T0;
#pragma unroll 1
    for (int k = 0; k < S.h; ++k) {   // both halves
        const M d = A[k * W];
        const M rd = d > T[k] ? M(1) / d : M(0);
        for (int q = lane; q < np; q += kBandCols) {   // A(k+1+u, k+1+v) -= A(k+1+u, k) A(k+1+v, k) / d
            const int u = tri_s[q] >> 8, v = tri_s[q] & 255;
            const M lu = A[(k + 1 + u) * W + u + 1] * rd;
            M *x = A + (k + 1 + u) * W + (u - v);
            *x = fma(-lu, A[(k + 1 + v) * W + v + 1], *x);
            if (v == 0) L[(k + 1 + u) * bw + u] = lu;
        }
        if (lane == 0) D[k] = rd;
        __syncwarp();
    }
    // the middle rows: half 1's share of them to half 0's, then on with half 0
    for (int q = t; q < S.s * W; q += 32) {
        const int u = q / W, d = q - u * W, v = u - d;
        if (v >= 0) A0[(S.h + u) * W + d] += A1[(S.h + S.s - 1 - v) * W + d];
    }
    __syncwarp();
#pragma unroll 1
    for (int k = S.h; k < S.rows; ++k) {
        const M d = A0[k * W];
        const M rd = d > T0[k] ? M(1) / d : M(0);
        const int m = S.rows - 1 - k < bw ? S.rows - 1 - k : bw, nm = m * (m + 1) / 2;
        for (int q = t; q < nm; q += 32) {
            const int u = tri_s[q] >> 8, v = tri_s[q] & 255;
            const M lu = A0[(k + 1 + u) * W + u + 1] * rd;
            M *x = A0 + (k + 1 + u) * W + (u - v);
            *x = fma(-lu, A0[(k + 1 + v) * W + v + 1], *x);
            if (v == 0) L0[(k + 1 + u) * bw + u] = lu;
        }
        if (t == 0) D0[k] = rd;
        __syncwarp();
    }
    const int col = blockIdx.x * kBandCols + lane;
    const bool live = col < n && (col < S.rows ? D0[col] : D1[n - 1 - col]) > M(0);
    if (bw <= 4) band_solve<M, 4>(S, L0, L1, D0, D1, Y, col, live);
    else if (bw <= 8) band_solve<M, 8>(S, L0, L1, D0, D1, Y, col, live);
    else if (bw <= 12) band_solve<M, 12>(S, L0, L1, D0, D1, Y, col, live);
    else band_solve<M, 25>(S, L0, L1, D0, D1, Y, col, live);
    if (col < n)
        for (int r = half; r < n; r += 2) inv[cell_s[r] * n + cell_s[col]] = Y[r * kBandCols + lane];
}

}  // namespace oscar
