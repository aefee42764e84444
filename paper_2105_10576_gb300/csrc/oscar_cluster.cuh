// Multigrid levels worked by one thread-block cluster (sm_103a).
//
// The lower levels of the V-cycle are far too small to fill the GPU, and as
// one launch per half sweep they are a chain of dependent launches (1.2 us
// each); in a single CTA they are bound by that SM's issue rate and, in FP64,
// by its two FP64 FMAs per clock. Here a cluster of up to 16 CTAs holds them
// in distributed shared memory: each CTA owns a slab of columns (an x range)
// of every level and works it with a wide margin of ghost columns. A cluster
// barrier takes 0.26-0.31 us (256-512 threads per CTA), a block barrier a
// quarter of that, so the ghosts are recomputed rather than exchanged: given
// the right-hand side on D ghost columns, each half sweep is valid on one
// column less, and a whole level (pre-smoothing, residual, prolongation,
// post-smoothing) passes with block barriers only. What crosses CTAs is the
// restricted right-hand side, once per level, stored into every CTA whose
// margin covers it (st.shared::cluster), followed by one cluster barrier.
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
    float rncol, rny, rhj;   // reciprocals for the cell decomposition
    const M *c[3], *idiag;
    // shared-memory byte offsets: x, b, reciprocal diagonal, low-face
    // coefficients per direction, colour lists (local indices by column), the
    // coarse local index of each colour-0 entry
    int ox, ob, oi, oc[3], ol[2], op;
};
template <typename M> struct ClLevels {
    int n, nc, lnc;          // levels, CTAs (a power of two) and their log2
    int cols;                // columns of the coarsest level
    int ors, obx, oinv;      // residual scratch, gathered right-hand side and inverse rows of the coarsest level
    int ored;                // reduction scratch
    const M *inv;            // explicit inverse of the coarsest level (row-major)
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
template <typename M> __device__ __forceinline__ int cl_start(const ClLevels<M> &P, const ClLevel<M> &L, int r) {
    return min(((r * P.cols) >> P.lnc) << L.sh, L.nx);
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

// store v into field f (a shared-memory array in the level's layout) at global
// column i, position m of the column, in every other CTA whose ghosts of depth
// d cover it
template <typename M>
__device__ __forceinline__ void cl_push(const ClLevels<M> &P, const ClLevel<M> &L, M *f, int i, int m, int d, int rank, M v) {
    for (int r = rank - 1; r >= 0; --r) {
        if (i >= cl_start(P, L, r + 1) + d) break;
        cl_store(cl_addr(f + (i - cl_start(P, L, r) + L.G) * L.ps + m, r), v);
    }
    for (int r = rank + 1; r < P.nc; ++r) {
        const int s = cl_start(P, L, r);
        if (i < s - d) break;
        cl_store(cl_addr(f + (i - s + L.G) * L.ps + m, r), v);
    }
}

// Coefficients and lists of every level into shared memory; x and b cleared.
// Ends without a barrier.
template <int DIM, typename M>
__device__ __forceinline__ void cl_load(const ClLevels<M> &P, unsigned char *sm, int rank) {
    const int t = threadIdx.x, nt = blockDim.x;
    for (int l = 0; l < P.n; ++l) {
        const ClLevel<M> &L = P.L[l];
        const int s = cl_start(P, L, rank);
        M *x = (M *)(sm + L.ox), *b = (M *)(sm + L.ob), *id = (M *)(sm + L.oi);
        M *c0 = (M *)(sm + L.oc[0]), *c1 = (M *)(sm + L.oc[1]), *c2 = (M *)(sm + L.oc[2]);
        for (int c = t; c < L.nloc; c += nt) { x[c] = M(0); b[c] = M(0); }
        const int pc = L.ps - L.ny * L.nz;   // unused cells at the end of a column
        for (int c = t; c < L.ncol * pc; c += nt) {
            const int q = c / pc, o = q * L.ps + L.ny * L.nz + c - q * pc;
            id[o] = c0[o] = c1[o] = M(0);
            if (DIM == 3) c2[o] = M(0);
        }
        for (int c = t; c < L.ncol * L.ny * L.nz; c += nt) {   // x fastest: rows of the global arrays
            int q, j, k;
            split3(c, L.ncol, L.rncol, L.ny, L.rny, q, j, k);
            const int i = s - L.G + q, o = q * L.ps + j + L.ny * k;
            M v0 = M(0), v1 = M(0), v2 = M(0), vi = M(0);
            if (i >= 0 && i < L.nx) {
                const int gc = i + L.nx * (j + L.ny * k);
                v1 = L.c[1][i + L.nx * (j + (L.ny + 1) * k)];
                if (DIM == 3) v2 = L.c[2][gc];
                vi = L.idiag[gc];
            }
            if (i >= 0 && i <= L.nx) v0 = L.c[0][i + (L.nx + 1) * (j + L.ny * k)];   // i = nx: the outlet, x = 0 beyond it
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
            int tj, k, q;
            split3(h, hj, L.rhj, L.nz, 1.0f / (float)L.nz, tj, k, q);
            const int i = s - L.G + q;
#pragma unroll
            for (int colour = 0; colour < 2; ++colour) {
                const int j = 2 * tj + ((i + k + colour) & 1);
                const bool in = i >= 0 && i < L.nx && j < L.ny;
                ((unsigned short *)(sm + L.ol[colour]))[h] = in ? (unsigned short)(q * L.ps + j + L.ny * k) : kClNone;
                if (colour == 0 && !last) {
                    const int qc = (i >> (L.rx >> 1)) - cs + C.G;
                    ((unsigned short *)(sm + L.op))[h] =
                        in && qc >= 0 && qc < C.ncol ? (unsigned short)(qc * C.ps + (j >> (L.ry >> 1)) + C.ny * (k >> (L.rz >> 1)))
                                                     : (unsigned short)0;
                }
            }
        }
    }
}

// rows of the coarsest level's inverse on which x is needed, in local cell
// order without the columns' padding; written by an earlier kernel
template <typename M>
__device__ __forceinline__ void cl_load_inverse(const ClLevels<M> &P, unsigned char *sm, int rank) {
    const ClLevel<M> &L = P.L[P.n - 1];
    const ClRange R = cl_range(P, L, rank, L.E);
    const int ne = L.nx * L.ny * L.nz, pl = L.ny * L.nz;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    M *inv = (M *)(sm + P.oinv);
    for (int row = warp; row < (R.q1 - R.q0) * pl; row += nw) {
        const int q = row / pl, m = row - q * pl;
        const M *src = P.inv + (size_t)(R.s - L.G + R.q0 + q + L.nx * m) * ne;
        for (int v = lane; v < ne; v += 32) inv[row * ne + v] = src[v];
    }
}

// sum of the neighbour terms of one row: one after the other (the order of
// mg_row_off), or the two of a direction first on the smallest levels
template <int DIM, typename M>
__device__ __forceinline__ M cl_off(const M *w, const M *x, int c, int ps, int ny, bool paired) {
    const M a0 = w[0] * x[c - ps], a1 = w[1] * x[c + ps];
    const M b0 = w[2] * x[c - 1], b1 = w[3] * x[c + 1];
    M off = a0 + a1;
    off = paired ? off + (b0 + b1) : (off + b0) + b1;
    if (DIM == 3) {
        const M d0 = w[4] * x[c - ny], d1 = w[5] * x[c + ny];
        off = paired ? off + (d0 + d1) : (off + d0) + d1;
    }
    return off;
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

// one colour of a red-black sweep on the slab and d columns beyond it (no barrier)
template <int DIM, typename M>
__device__ __forceinline__ void cl_sweep(const ClLevels<M> &P, const ClLevel<M> &L, unsigned char *sm, int colour, int d,
                                         int rank) {
    M *x = (M *)(sm + L.ox);
    const M *b = (const M *)(sm + L.ob), *id = (const M *)(sm + L.oi);
    const unsigned short *lst = (const unsigned short *)(sm + L.ol[colour]);
    const ClRange R = cl_range(P, L, rank, d);
    for (int h = R.q0 * L.ce + threadIdx.x; h < R.q1 * L.ce; h += blockDim.x) {
        const int c = lst[h];
        if (c == kClNone) continue;
        M w[2 * DIM];
        cl_row<DIM, M>(L, sm, c, w);
        x[c] = (b[c] + cl_off<DIM, M>(w, x, c, L.ps, L.ny, L.paired)) * id[c];
    }
}
// the first colour-0 half sweep from x = 0, on every column that holds b
template <typename M>
__device__ __forceinline__ void cl_first_sweep(const ClLevels<M> &P, const ClLevel<M> &L, unsigned char *sm, int rank) {
    M *x = (M *)(sm + L.ox);
    const M *b = (const M *)(sm + L.ob), *id = (const M *)(sm + L.oi);
    const unsigned short *lst = (const unsigned short *)(sm + L.ol[0]);
    const ClRange R = cl_range(P, L, rank, L.G);
    for (int h = R.q0 * L.ce + threadIdx.x; h < R.q1 * L.ce; h += blockDim.x) {
        const int c = lst[h];
        if (c != kClNone) x[c] = b[c] * id[c];
    }
}

// residual of the slab's cells, then b of the next level = the sum over the
// children (x fastest), stored into every CTA whose ghosts cover it (on the
// coarsest level, into every CTA's gathered copy)
template <int DIM, typename M>
__device__ __forceinline__ void cl_restrict(const ClLevels<M> &P, int l, unsigned char *sm, int rank) {
    const ClLevel<M> &L = P.L[l], &C = P.L[l + 1];
    M *rs = (M *)(sm + P.ors);
    const ClRange F = cl_range(P, L, rank, 0);
    {
        const M *x = (const M *)(sm + L.ox), *b = (const M *)(sm + L.ob);
        const unsigned short *l0 = (const unsigned short *)(sm + L.ol[0]), *l1 = (const unsigned short *)(sm + L.ol[1]);
        const int n = F.w * L.ce;
        for (int h = threadIdx.x; h < 2 * n; h += blockDim.x) {
            const int c = h < n ? l0[F.q0 * L.ce + h] : l1[F.q0 * L.ce + h - n];
            if (c == kClNone) continue;
            M w[2 * DIM], dg = M(0);
            cl_row<DIM, M>(L, sm, c, w);
#pragma unroll
            for (int a = 0; a < DIM; ++a) dg += w[2 * a] + w[2 * a + 1];   // the diagonal as it was formed
            rs[c - F.q0 * L.ps] = b[c] - (dg * x[c] - cl_off<DIM, M>(w, x, c, L.ps, L.ny, L.paired));
        }
    }
    __syncthreads();
    const ClRange S = cl_range(P, C, rank, 0);
    const bool last = l + 1 == P.n - 1;
    M *bc = (M *)(sm + C.ob), *bx = (M *)(sm + P.obx);
    const float rw = 1.0f / (float)S.w;
    for (int q = threadIdx.x; q < S.w * C.ny * C.nz; q += blockDim.x) {
        int p, J, K;
        split3(q, S.w, rw, C.ny, C.rny, p, J, K);
        M acc = M(0);
        for (int kk = K * L.rz; kk < min((K + 1) * L.rz, L.nz); ++kk)
            for (int jj = J * L.ry; jj < min((J + 1) * L.ry, L.ny); ++jj)
                for (int pp = p * L.rx; pp < min((p + 1) * L.rx, F.w); ++pp) acc += rs[pp * L.ps + jj + L.ny * kk];
        const int i = S.s + p;
        if (last) {
            const int gc = i + C.nx * (J + C.ny * K);
            for (int r = 0; r < P.nc; ++r) cl_store(cl_addr(bx + gc, r), acc);
        } else {
            const int m = J + C.ny * K;
            bc[(p + C.G) * C.ps + m] = acc;
            cl_push(P, C, bc, i, m, C.G, rank, acc);
        }
    }
}

// x = inverse * b on the coarsest level, on the columns that need it: a warp
// per row, lanes over the columns of the inverse, four rows at a time
template <typename M> __device__ __forceinline__ void cl_exact(const ClLevels<M> &P, unsigned char *sm, int rank) {
    const ClLevel<M> &L = P.L[P.n - 1];
    const ClRange R = cl_range(P, L, rank, L.E);
    const int ne = L.nx * L.ny * L.nz, pl = L.ny * L.nz, nr = (R.q1 - R.q0) * pl;
    const M *inv = (const M *)(sm + P.oinv), *bx = (const M *)(sm + P.obx);
    M *x = (M *)(sm + L.ox);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int r0 = warp; r0 < nr; r0 += 4 * nw) {
        M acc[4] = {M(0), M(0), M(0), M(0)};
        for (int m = lane; m < ne; m += 32) {
            const M v = bx[m];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (r0 + u * nw < nr) acc[u] += inv[(r0 + u * nw) * ne + m] * v;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (r0 + u * nw < nr) acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], o);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int row = r0 + u * nw, q = row / pl;
            if (lane == 0 && row < nr) x[(R.q0 + q) * L.ps + row - q * pl] = acc[u];
        }
    }
}

// x of the colour-0 cells += the coarser level's x
template <typename M> __device__ __forceinline__ void cl_prolong(const ClLevels<M> &P, int l, unsigned char *sm, int rank) {
    const ClLevel<M> &L = P.L[l];
    M *x = (M *)(sm + L.ox);
    const M *xc = (const M *)(sm + P.L[l + 1].ox);
    const unsigned short *lst = (const unsigned short *)(sm + L.ol[0]), *par = (const unsigned short *)(sm + L.op);
    const ClRange R = cl_range(P, L, rank, L.E + 2 * L.nu);
    for (int h = R.q0 * L.ce + threadIdx.x; h < R.q1 * L.ce; h += blockDim.x) {
        const int c = lst[h];
        if (c != kClNone) x[c] += xc[par[h]];
    }
}

// The V-cycle over the cluster's levels. On entry the first level's b (with
// its ghosts; the gathered b when it is the coarsest) is in place and a
// cluster barrier has been passed since. On return x of the first level is
// valid on E columns beyond the slab; no barrier has been passed since its
// last half sweep (the solution, when it is the coarsest level).
template <int DIM, typename M>
__device__ __forceinline__ void cl_vcycle(const ClLevels<M> &P, unsigned char *sm, int rank) {
    for (int l = 0; l < P.n - 1; ++l) {
        const ClLevel<M> &L = P.L[l];
        cl_first_sweep<M>(P, L, sm, rank);
        __syncthreads();
        for (int s = 0; s < L.nu; ++s) {
            if (s > 0) {
                cl_sweep<DIM, M>(P, L, sm, 0, L.D - 2 * s, rank);
                __syncthreads();
            }
            // the last one is read by the residual only
            cl_sweep<DIM, M>(P, L, sm, 1, s == L.nu - 1 ? 1 : L.D - 2 * s - 1, rank);
            __syncthreads();
        }
        cl_restrict<DIM, M>(P, l, sm, rank);
        cl_sync(P.nc);
    }
    cl_exact<M>(P, sm, rank);
    for (int l = P.n - 2; l >= 0; --l) {
        const ClLevel<M> &L = P.L[l];
        __syncthreads();
        cl_prolong<M>(P, l, sm, rank);
        for (int s = 0; s < L.nu; ++s) {
            __syncthreads();
            cl_sweep<DIM, M>(P, L, sm, 1, L.E + 2 * (L.nu - s) - 1, rank);
            __syncthreads();
            cl_sweep<DIM, M>(P, L, sm, 0, L.E + 2 * (L.nu - s) - 2, rank);
        }
    }
}

// The V-cycle below the per-level kernels: b of the first level from b_top,
// its x to x_top. Coefficients (fixed during a solve) are loaded before the
// grid-dependency wait.
template <int DIM, typename M>
__global__ void __launch_bounds__(512, 1) k_mg_cluster(ClLevels<M> P, const M *__restrict__ b_top, M *__restrict__ x_top) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int rank = cl_rank();
    const ClLevel<M> &L = P.L[0];
    cl_load<DIM, M>(P, sm, rank);
    cl_load_inverse<M>(P, sm, rank);
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
    double alpha, beta;
    float alpha_f, beta_f;
    int more;
};

// totals over the cluster of nv FP64 values per thread, valid in warp 0 of
// every CTA (same order everywhere: same result). Two buffers, alternating: a
// CTA may store for the next reduction while another still reads this one.
template <typename M>
__device__ __forceinline__ void cl_sum(const ClLevels<M> &P, unsigned char *sm, int rank, int &buf, double *v, int nv) {
    double *sh = (double *)(sm + P.ored), *slot = sh + 512 + buf * 4 * kMaxCluster;
    const int t = threadIdx.x, nt = blockDim.x;
    for (int q = 0; q < nv; ++q) {
        __syncthreads();
        sh[t] = v[q];
        __syncthreads();
        if (t < 32) {
            double s = sh[t];
            for (int m = t + 32; m < nt; m += 32) s += sh[m];
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (t < P.nc) cl_store(cl_addr(slot + q * kMaxCluster + rank, t), s);
        }
    }
    cl_sync(P.nc);
    if (t < 32)
        for (int q = 0; q < nv; ++q) {
            double s = t < P.nc ? slot[q * kMaxCluster + t] : 0.0;
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            v[q] = s;
        }
    buf ^= 1;
}
// the same for one value of the vectors' type: FP64 as above, FP32 in
// compensated pairs; the total is valid in thread 0
template <typename M>
__device__ __forceinline__ double cl_dot(const ClLevels<M> &P, unsigned char *sm, int rank, int &buf, DotAcc64 a) {
    cl_sum(P, sm, rank, buf, &a.s, 1);
    return a.s;
}
template <typename M>
__device__ __forceinline__ double cl_dot(const ClLevels<M> &P, unsigned char *sm, int rank, int &buf, DotAcc32 a) {
    float2 *slot = (float2 *)((double *)(sm + P.ored) + 512 + buf * 4 * kMaxCluster);
    const int t = threadIdx.x;
    float s = a.s, e = a.e;
    block_pair_f(s, e);
    if (t < 32) {
        s = __shfl_sync(0xffffffffu, s, 0);
        e = __shfl_sync(0xffffffffu, e, 0);
        if (t < P.nc) {
            const unsigned d = cl_addr(slot + rank, t);
            cl_store(d, s);
            cl_store(d + 4, e);
        }
    }
    cl_sync(P.nc);
    double tot = 0.0;
    if (t < 32) {
        s = t < P.nc ? slot[t].x : 0.f;
        e = t < P.nc ? slot[t].y : 0.f;
        warp_sum_pair(s, e);
        if (t == 0) tot = (double)s + (double)e;
    }
    buf ^= 1;
    return tot;
}

// own cells of level 0: own column pc, row j, x fastest (rows of the global arrays)
#define CL_OWN_CELLS()                                                                                        \
    for (int g_ = t, pc, j, k_; g_ < S.w * L.ny && (split3(g_, S.w, rw, L.ny, L.rny, pc, j, k_), true); g_ += blockDim.x)

// groups of own cells that one thread of the launched CG kernels sums
// (launch_rpt): own column pc, rows j0 + u by for u < rpt
#define CL_ROW_GROUPS(rpt)                                                                               \
    for (int g_ = t, nb_ = (L.ny + A.by * (rpt) - 1) / (A.by * (rpt)), pc, ty_, blk_; g_ < S.w * A.by * nb_; \
         g_ += blockDim.x)                                                                               \
        if (split3(g_, A.by, rby, nb_, 1.0f / (float)nb_, ty_, blk_, pc); true)                          \
            if (const int j0 = blk_ * A.by * (rpt) + ty_; j0 < L.ny)

template <typename T>
__global__ void __launch_bounds__(512, 1) k_solve_cluster(ClLevels<T> P, ClSolve A) {
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ ClControl K;
    constexpr bool MIXED = sizeof(T) == sizeof(float);
    const int rank = cl_rank(), t = threadIdx.x;
    const ClLevel<T> &L = P.L[0];
    const int ps = L.ps;
    const ClRange S = cl_range(P, L, rank, 0);
    cl_load<2, T>(P, sm, rank);
    cl_load_inverse<T>(P, sm, rank);
    T *x = (T *)(sm + L.ox), *r = (T *)(sm + L.ob), *bx = (T *)(sm + P.obx);
    T *p = (T *)(sm + A.op) - (L.G - 1) * ps, *Ap = (T *)(sm + A.oap) - (L.G - 1) * ps, *e = (T *)(sm + A.oe) - (L.G - 1) * ps;
    for (int c = t + (L.G - 1) * ps; c < (L.G + S.w + 1) * ps; c += blockDim.x) { p[c] = T(0); Ap[c] = T(0); }
    const float rw = 1.0f / (float)S.w, rby = 1.0f / (float)A.by;
    int buf = 0, its = 0, outer = 0, nan_seen = 0, notconv = 0;
    cl_sync(P.nc);   // every CTA's shared memory is ready for remote stores
    griddep_wait();

    // residual of an own cell, with the copies the ghosts (or, when level 0 is
    // the coarsest, the gathered right-hand side) need
    auto put_r = [&](int pc, int j, T rc) {
        r[(pc + L.G) * ps + j] = rc;
        if (P.n == 1)
            for (int m = 0; m < P.nc; ++m) cl_store(cl_addr(bx + S.s + pc + L.nx * j, m), rc);
        else
            cl_push(P, L, r, S.s + pc, j, L.G, rank, rc);
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
                const int tp = g / L.ny, j = g - tp * L.ny, lo = (2 * tp + L.G) * ps + j, odd = (S.s + j) & 1;
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
                K.beta = K.rz0 != 0.0 ? rz / K.rz0 : 0.0;
                K.beta_f = (float)K.beta;
            }
            __syncthreads();
            typename DotAcc<T>::type dp;
            const T *c0 = (const T *)(sm + L.oc[0]), *c1 = (const T *)(sm + L.oc[1]);
            if constexpr (MIXED) {   // p = z + beta p, Ap = M z + beta Ap, p.Ap
                const T be = K.beta_f;
                const bool fresh = be == T(0);
                CL_ROW_GROUPS(kApplyRows) {
                    T a = T(0);
#pragma unroll
                    for (int u = 0; u < kApplyRows; ++u) {
                        const int j = j0 + u * A.by;
                        if (j >= L.ny) break;
                        const int c = (pc + L.G) * ps + j;
                        const T zc = x[c];
                        const T pn = fresh ? zc : zc + be * p[c];
                        T y = c0[c] * (zc - x[c - ps]);
                        y += c0[c + ps] * (zc - x[c + ps]);
                        y += c1[c] * (zc - x[c - 1]);
                        y += c1[c + 1] * (zc - x[c + 1]);
                        const T an = fresh ? y : y + be * Ap[c];
                        p[c] = pn;
                        Ap[c] = an;
                        a += pn * an;
                    }
                    dp.add(a);
                }
            } else {   // p = z + beta p (one ghost column as well), Ap = M p, p.Ap
                const T be = K.beta;
                for (int c = t + (L.G - 1) * ps; c < (L.G + S.w + 1) * ps; c += blockDim.x) p[c] = x[c] + be * p[c];
                __syncthreads();
                CL_ROW_GROUPS(1) {
                    const int c = (pc + L.G) * ps + j0;
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
            CL_ROW_GROUPS(kUpdateRows) {   // x += alpha p, r -= alpha Ap, r.r
                T a = T(0);
#pragma unroll
                for (int u = 0; u < kUpdateRows; ++u) {
                    const int j = j0 + u * A.by;
                    if (j >= L.ny) break;
                    const int c = (pc + L.G) * ps + j;
                    if constexpr (MIXED) e[c] = it == 0 ? al * p[c] : e[c] + al * p[c];
                    else A.q[S.s + pc + L.nx * j] += al * p[c];
                    const T rc = r[c] - al * Ap[c];
                    put_r(pc, j, rc);
                    a += rc * rc;
                }
                dr.add(a);
            }
            const double rr = cl_dot(P, sm, rank, buf, dr);
            ++it;
            ++its;
            if (t == 0) {
                K.rz0 = K.rz1;
                const double rn = sqrt(rr);
                const bool bad = !isfinite(rn);
                nan_seen |= bad;
                bool more = !bad && rn > (MIXED ? K.itarget : K.target);
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
                cl_push(P, L, x, S.s + pc, j, 1, rank, e[c]);
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
// after it (ctl[C_PACK] counts them); in between the stored inverse is kept (a
// preconditioner component: a stale one changes iterations, not the solution).
__device__ __forceinline__ bool inverse_due(int *ctl, int refresh) {
    __shared__ int due_s;
    if (threadIdx.x == 0) {
        due_s = ctl[C_PACK] % refresh == 0;
        ctl[C_PACK] += 1;
    }
    __syncthreads();
    return due_s;
}

// FP32: Gauss-Jordan elimination without pivoting, in place (the matrix is
// symmetric positive definite: the fluid is connected to the Dirichlet
// outlet). Rows of cells that are solid or have no coefficients decouple; a
// pivot that vanishes (a pocket cut off from the outlet) drops its row and
// column. Each thread keeps an 8x8 tile in registers; per pivot its row and
// column pass through double-buffered shared memory, one block barrier per
// pivot (128 pivots, against two barriers and 48 shared-memory accesses per
// thread and pivot for a matrix in shared memory). Every entry sees the same
// operations in the same order whatever the layout.
constexpr int kGjThreads = 256, kGjTile = 8;
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
template <int DIM>
__global__ void __launch_bounds__(kGjThreads) k_mg_inverse_dense(GridD g, MG3<float> cc, const float *__restrict__ diag,
                                                                 const uint8_t *__restrict__ fluid,
                                                                 float *__restrict__ inv, int refresh,
                                                                 int *__restrict__ ctl) {
    static_assert(kGjThreads * kGjTile * kGjTile == kExactCells * kExactCells, "tiles cover the matrix");
    constexpr int B = kGjTile, TC = kExactCells / B;
    griddep_wait();
    if (!inverse_due(ctl, refresh)) return;
    __shared__ __align__(16) float rowb[2][kExactCells], colb[2][kExactCells];
    const int t = threadIdx.x, n = g.ncell, i0 = (t / TC) * B, j0 = (t % TC) * B;
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
    // publish row and column k of the current matrix
    auto publish = [&](int k) {
        float *rb = rowb[k & 1], *cb = colb[k & 1];
        const int ku = k - i0, kv = k - j0;
        if (ku >= 0 && ku < B)
            static_for<B>([&](auto v) {
                float a = 0.f;
                static_for<B>([&](auto u) { a = ku == u ? A[u * B + v] : a; });
                rb[j0 + v] = a;
            });
        if (kv >= 0 && kv < B)
            static_for<B>([&](auto u) {
                float a = 0.f;
                static_for<B>([&](auto v) { a = kv == v ? A[u * B + v] : a; });
                cb[i0 + u] = a;
            });
    };
    publish(0);
    for (int k = 0; k < n; ++k) {
        __syncthreads();
        const float *rb = rowb[k & 1], *cb = colb[k & 1];
        const float pv = rb[k];
        const bool skip = !(pv > 0.f);
        const float pinv = skip ? 0.f : 1.f / pv;
        float nk[B], ai[B];
        static_for<B>([&](auto v) {
            nk[v] = rb[j0 + v] * pinv;   // the normalised pivot row
            ai[v] = cb[i0 + v];
        });
        const int ku = k - i0, kv = k - j0;
        if (!skip) static_for<B * B>([&](auto q) { A[q] = fmaf(-ai[q / B], nk[q % B], A[q]); });
        if (kv >= 0 && kv < B)
            static_for<B * B>([&](auto q) { A[q] = q % B == kv ? (skip ? 0.f : -ai[q / B] * pinv) : A[q]; });
        if (ku >= 0 && ku < B)
            static_for<B * B>([&](auto q) {
                A[q] = q / B == ku ? (skip ? 0.f : (q % B == kv ? pinv : nk[q % B])) : A[q];
            });
        if (k + 1 < n) publish(k + 1);
    }
    static_for<B * B>([&](auto q) {
        if (i0 + q / B < n && j0 + q % B < n) inv[(i0 + q / B) * n + j0 + q % B] = A[q];
    });
}

// FP64: LDL^T without pivoting in band form (the matrix is symmetric positive
// definite: the fluid is connected to the Dirichlet outlet), cells ordered
// with the shortest axis fastest, so that the band is the product of the two
// shortest extents (4 to about 25 for at most 128 cells), then one thread per
// column of the inverse solves L D L^T x = e_j: n^2 (2 bw + 1) operations
// instead of the n^3 of a dense elimination. Rows of cells that are solid or
// have no coefficients, and of pivots that vanish (a pocket cut off from the
// outlet), give a zero row and column. (A dense elimination is bound by the
// SM's two FP64 FMAs per clock: 1.1 ms at 128 cells.)
template <int DIM, typename M>
__global__ void __launch_bounds__(128) k_mg_inverse_band(GridD g, MG3<M> cc, const M *__restrict__ diag,
                                                    const uint8_t *__restrict__ fluid, M *__restrict__ inv, int refresh,
                                                    int *__restrict__ ctl) {
    extern __shared__ __align__(16) unsigned char sm[];
    griddep_wait();
    if (!inverse_due(ctl, refresh)) return;
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
    M *B = (M *)sm;                       // B[r W + d] = A(r, r - d), then L (d > 0) and D (d = 0)
    M *Y = B + (size_t)kExactCells * W;   // Y[i n + j]: column j of the inverse, band order
    __shared__ int cell_s[kExactCells];   // cell of a band index
    for (int q = t; q < n * W; q += blockDim.x) B[q] = M(0);
    __syncthreads();
    for (int c = t; c < n; c += blockDim.x) {
        const int i = c % g.nx, j = (c / g.nx) % g.ny, k = c / (g.nx * g.ny);
        const int r = i * st[0] + j * st[1] + k * st[2];
        cell_s[r] = c;
        const M d = diag[c];
        const bool live = fluid[c] && d > M(0);
        if (!live) continue;
        B[r * W] = d;
        const int ijk[3] = {i, j, k};
#pragma unroll
        for (int a = 0; a < DIM; ++a)   // the low neighbours are those of smaller band index
            if (ijk[a] > 0) B[r * W + st[a]] = -cc.a[a][flo(g, a, i, j, k)];
    }
    // right-looking factorisation: after step k the columns beyond k hold the Schur complement
    for (int k = 0; k < n; ++k) {
        __syncthreads();
        const M d = B[k * W];
        const bool ok = d > M(0);
        const M rd = ok ? M(1) / d : M(0);
        const int m = min(bw, n - 1 - k);
        for (int q = t; q < m * m; q += blockDim.x) {   // A(k+1+u, k+1+v) -= A(k+1+u, k) A(k+1+v, k) / d, v <= u
            const int u = q / m, v = q - u * m;
            if (v > u) continue;
            B[(k + 1 + u) * W + (u - v)] -= B[(k + 1 + u) * W + u + 1] * rd * B[(k + 1 + v) * W + v + 1];
        }
    }
    __syncthreads();
    // column k of L: A(r, k) / D(k); a vanished pivot drops its row and column
    for (int q = t; q < n * bw; q += blockDim.x) {
        const int r = q / bw, d = q - r * bw + 1;
        if (r < d) continue;
        const M p = B[(r - d) * W];
        B[r * W + d] = p > M(0) ? B[r * W + d] / p : M(0);
    }
    __syncthreads();
    if (t < n) {
        const M dt = B[t * W];
        for (int i = 0; i < t; ++i) Y[i * n + t] = M(0);
        for (int i = t; i < n; ++i) {   // L y = e_t
            M a0 = i == t ? M(1) : M(0), a1 = M(0);
            const int m = min(bw, i - t);
            int d = 1;
            for (; d + 1 <= m; d += 2) {
                a0 = fma(-B[i * W + d], Y[(i - d) * n + t], a0);
                a1 = fma(-B[i * W + d + 1], Y[(i - d - 1) * n + t], a1);
            }
            if (d <= m) a0 = fma(-B[i * W + d], Y[(i - d) * n + t], a0);
            Y[i * n + t] = a0 + a1;
        }
        for (int i = n - 1; i >= 0; --i) {   // L^T x = D^-1 y
            const M di = B[i * W];
            M a0 = di > M(0) ? Y[i * n + t] / di : M(0), a1 = M(0);
            const int m = min(bw, n - 1 - i);
            int d = 1;
            for (; d + 1 <= m; d += 2) {
                a0 = fma(-B[(i + d) * W + d], Y[(i + d) * n + t], a0);
                a1 = fma(-B[(i + d + 1) * W + d + 1], Y[(i + d + 1) * n + t], a1);
            }
            if (d <= m) a0 = fma(-B[(i + d) * W + d], Y[(i + d) * n + t], a0);
            const bool live = di > M(0) && dt > M(0);
            Y[i * n + t] = live ? a0 + a1 : M(0);
        }
    }
    __syncthreads();
    for (int q = t; q < n * n; q += blockDim.x) {
        const int r = q / n, j = q - r * n;
        inv[cell_s[r] * n + cell_s[j]] = Y[q];
    }
}

}  // namespace oscar
