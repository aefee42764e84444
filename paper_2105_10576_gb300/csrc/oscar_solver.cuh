// Orchestration of the OSCAR steps (Maes & Menke, arXiv 2105.10576,
// Sections 2.2, 3.1, 3.2) as CUDA graphs.
//
// Each API call (drag step, relaxation, standard step) launches one
// instantiated graph and synchronises once. Inside the graph a pressure solve
// is one conditional WHILE node of PCG iterations, whose last kernel (k_cg_check
// in FP64, k_cg_refine on the mixed path, which also ends the FP64
// defect-correction trips) decides on the next one; a small 2D grid's solve is
// one launch of k_solve_cluster, without a loop node. The relaxation is an outer
// WHILE node whose last reduction applies the paper's early exit (E_k < tol or
// k = N) on the device. Dot products of FP32 vectors are summed in compensated
// pairs. Graphs are captured from the same launch sequence the eager mode
// issues, and rebuilt when the time step changes.
#pragma once
#include <stdlib.h>
#include <string.h>

#include "oscar_cluster.cuh"

namespace oscar {

#define OSCAR_LAUNCH_CHECK()                                                                              \
    do {                                                                                                  \
        cudaError_t e_ = cudaGetLastError();                                                              \
        if (e_ != cudaSuccess) {                                                                          \
            fprintf(stderr, "oscar: CUDA error %s at %s:%d\n", cudaGetErrorString(e_), __FILE__, __LINE__); \
            return OSCAR_E_CUDA;                                                                          \
        }                                                                                                 \
    } while (0)

#define OSCAR_TRY(x)              \
    do {                          \
        int rc_ = (x);            \
        if (rc_) return rc_;      \
    } while (0)

inline int nblk(long long n) { return (int)((n + BS - 1) / BS); }

// Kernel launch with programmatic stream serialization: the next kernel's
// launch overlaps the tail of this one (each kernel waits in griddep_wait()).
// nc > 1: a cluster of that many CTAs. pdl = false: full dependencies (the
// first kernel after a fork or a join of streams).
template <typename... KArgs, typename... Args>
inline void launchx(bool pdl, int nc, void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                    Args &&...args) {
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    int na = 0;
    if (pdl) {
        attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[na++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (nc > 1) {
        attr[na].id = cudaLaunchAttributeClusterDimension;
        attr[na].val.clusterDim.x = (unsigned)nc;
        attr[na].val.clusterDim.y = attr[na].val.clusterDim.z = 1;
        ++na;
    }
    cfg.attrs = attr;
    cfg.numAttrs = na;
    if (Profiler *P = t_prof) {   // in-step timing (eager steps only; never while capturing)
        int slot = prof_begin(P, st, (const void *)kern, grid, block);
        cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
        prof_end(P, st, slot);
    } else {
        cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
    }
}
template <typename... KArgs, typename... Args>
inline void launchk(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args &&...args) {
    launchx(true, 1, kern, grid, block, smem, st, std::forward<Args>(args)...);
}

// ---------------------------------------------------------------------------
// control kernel (one thread). The other loop decisions are taken by the
// finishing block of the reductions (see k_cg_init, k_cg_check, k_cg_refine,
// k_relax_accum).
// ---------------------------------------------------------------------------
static __global__ void k_relax_init(int *ctl, cudaGraphConditionalHandle h) {
    griddep_wait(); set_cond(ctl, h, ctl[C_N] > 0); }

// ---------------------------------------------------------------------------
// capture helpers
// ---------------------------------------------------------------------------
inline int cond_handle(Instance &I, cudaGraphConditionalHandle *h) {
    if (!I.capturing) { *h = 0; return 0; }
    cudaStreamCaptureStatus st;
    cudaGraph_t g;
    if (cudaStreamGetCaptureInfo(I.stream, &st, nullptr, &g, nullptr, nullptr, nullptr) != cudaSuccess ||
        st != cudaStreamCaptureStatusActive)
        return OSCAR_E_CUDA;
    if (cudaGraphConditionalHandleCreate(h, g, 0, 0) != cudaSuccess) return OSCAR_E_CUDA;
    return 0;
}

// Append a WHILE node at the capture point of I.stream and redirect I.stream
// to capture its body.
inline int begin_while(Instance &I, cudaGraphConditionalHandle h, cudaStream_t *saved) {
    cudaStreamCaptureStatus st;
    cudaGraph_t g;
    const cudaGraphNode_t *deps = nullptr;
    const cudaGraphEdgeData *ed = nullptr;
    size_t nd = 0;
    if (cudaStreamGetCaptureInfo(I.stream, &st, nullptr, &g, &deps, &ed, &nd) != cudaSuccess ||
        st != cudaStreamCaptureStatusActive)
        return OSCAR_E_CUDA;
    // cudaGraphNodeParams has no default constructor in C++: zero-initialised storage
    alignas(cudaGraphNodeParams) unsigned char buf[sizeof(cudaGraphNodeParams)];
    memset(buf, 0, sizeof(buf));
    cudaGraphNodeParams &np = *reinterpret_cast<cudaGraphNodeParams *>(buf);
    np.type = cudaGraphNodeTypeConditional;
    np.conditional.handle = h;
    np.conditional.type = cudaGraphCondTypeWhile;
    np.conditional.size = 1;
    cudaGraphNode_t node;
    if (cudaGraphAddNode(&node, g, deps, ed, nd, &np) != cudaSuccess) return OSCAR_E_CUDA;
    if (cudaStreamUpdateCaptureDependencies(I.stream, &node, nullptr, 1, cudaStreamSetCaptureDependencies) !=
        cudaSuccess)
        return OSCAR_E_CUDA;
    if (I.depth + 1 >= 4) return OSCAR_E_CUDA;
    cudaStream_t side = I.side[++I.depth];
    if (cudaStreamBeginCaptureToGraph(side, np.conditional.phGraph_out[0], nullptr, nullptr, 0,
                                      cudaStreamCaptureModeRelaxed) != cudaSuccess)
        return OSCAR_E_CUDA;
    *saved = I.stream;
    I.stream = side;
    return 0;
}

inline int end_while(Instance &I, cudaStream_t saved) {
    cudaGraph_t body;
    cudaError_t e = cudaStreamEndCapture(I.stream, &body);
    I.stream = saved;
    --I.depth;
    return e == cudaSuccess ? 0 : OSCAR_E_CUDA;
}

// Read the control words back (eager mode only).
inline int read_ctl(Instance &I) {
    if (cudaMemcpyAsync(I.ctl_host, I.ctl, C_COUNT * sizeof(int), cudaMemcpyDeviceToHost, I.stream) != cudaSuccess)
        return OSCAR_E_CUDA;
    return sync_bounded(I.stream, kSyncTimeoutSec);
}

// while (ctl[C_COND]) body(): a conditional WHILE node when capturing, a host
// loop (one read-back per trip) in eager mode. The decision is written by the
// kernel issued just before the loop and by the last kernel of the body.
template <class F> int loop_while(Instance &I, cudaGraphConditionalHandle h, F body) {
    if (I.capturing) {
        cudaStream_t saved;
        int rc = begin_while(I, h, &saved);
        if (rc) return rc;
        rc = body();
        int rc2 = end_while(I, saved);
        return rc ? rc : rc2;
    }
    for (;;) {
        int rc = read_ctl(I);
        if (rc) return rc;
        if (!I.ctl_host[C_COND]) return 0;
        rc = body();
        if (rc) return rc;
    }
}

// Which levels and grids go to a cluster, and of how many CTAs. The V-cycle's
// cluster takes levels of at most vcycle_cells x cta_cells cells (default 8192
// in FP32, where a launch per half sweep is still bound by its latency; in FP64
// the cluster is bound by FP64 issue above 1024 cells), of which a CTA works at
// most kVcycleRows. A 2D grid of at most kSolveCells is solved whole in one
// cluster when its vectors fit the shared memory and its slabs start at even
// columns (r.z pairs the columns 2 i and 2 i + 1; grids of one level, at most 128
// cells, have slabs of any width and go by launches, nx = 1 apart). Beyond that
// a solve alone is still shorter in the cluster (512x64 mixed 3.55 against 4.30
// ms per five steps, 5.90 launched without any cluster), but it holds 16 SMs for
// work that the launches spread thinner, and instances stepped together wait for
// each other (ten of 1024x128 to 128x16: 12.4 against 10.2 ms; 64: 392 against
// 419 M cell-updates/s).
constexpr int kSolveCells = 16384;
constexpr int kVcycleThreads = 512;
// CTAs of the V-cycle's cluster: at most 8. 16 make a V-cycle 1 to 2 us
// shorter, but all CTAs of a cluster need their SMs at the same time within one
// GPU processing cluster, and instances stepped together wait for it. One alone
// with 16 and 8: 1024x128 5.12 and 5.24 ms, 97x51x45 13.8 and 14.0, 256x64x64
// 21.7 and 21.8; together: ten of 1024x128 to 128x16 10.2 and 9.2 ms, 24 of
// 128x32x32 66.8 and 63.0 (before there were clusters 63.3), a mix of 36 in 2D
// and 3D 88.9 and 83.2 (83.3).
constexpr int kVcycleCtas = 8;
// Rows of the cluster's largest level that one CTA works, ghosts included: two
// of each colour per thread. The CTAs are bounded by the columns of the
// coarsest level, so on grids that are not long in x the level is worked by few
// of them, or by each of them almost whole, and the launches are shorter. us per
// PCG iteration with the level in the cluster and without: 4096 rows 16x1024
// 55.1 and 51.1, 64x64x64 75.6 and 72.5, 32x32x32 53.2 and 50.4; 2000 to 3000
// 120x48x48 76.3 and 74.9, 48x96x96 122.6 and 120.3, but 128x96x96 134.8 and
// 135.9, 100x600 57.7 and 58.1; 2048 64x128x128 130.9 and 129.8, 64x512 55.1 and
// 57.8; fewer 256x64x64 162.0 and 162.9, 1024x128 65.3 and 68.4.
constexpr int kVcycleRows = 4 * kVcycleThreads;
// fewer threads make the block and cluster barriers shorter, more take larger
// slabs with fewer entries per thread (128x16 FP64: 256 threads 8.03 ms per
// pass, 512 8.53; 512x64 mixed solved whole: 4.25 and 3.64)
inline int solve_threads(int ncell) { return ncell <= 8192 ? 256 : 512; }
// CTAs of the cluster: fewer exchange less, more have shorter slabs. FP32 at
// 128x16 (six sub-steps): 8 CTAs 2.48 ms, 16 2.55; at 211x26 3.92 and 3.56.
// FP64, bound by the SM's FP64 rate: 128x16 4.74 and 4.52. Many instances
// together are faster with 8 (64 of 256x32, mixed: 24.3 ms per step, with 16
// 27.1, before there were clusters 44.7).
template <typename T> inline int solve_ctas(int ncell) { return sizeof(T) == sizeof(float) && ncell <= 2048 ? 8 : 16; }
template <typename T> struct ClRule;
template <> struct ClRule<float> {
    static constexpr long long vcycle_cells = 8;
};
template <> struct ClRule<double> {
    static constexpr long long vcycle_cells = 1;
};

template <typename T> struct Impl {
    using M = T;
    using V = T;
    static T *tp(void *p) { return (T *)p; }
    static C3<T> c3(void *const *p) { C3<T> r; for (int a = 0; a < 3; ++a) r.a[a] = (const T *)p[a]; return r; }
    static C3<double> w64(const Instance &I) {
        C3<double> r;
        for (int a = 0; a < 3; ++a) r.a[a] = I.cf64[a];
        return r;
    }
    // FP64 copy of the level-0 coefficients of direction a (mixed path only)
    static double *cf64_out(Instance &I, int a) { return sizeof(T) == sizeof(double) ? nullptr : I.cf64[a]; }
    static P3<T> p3(void *const *p) { P3<T> r; for (int a = 0; a < 3; ++a) r.a[a] = (T *)p[a]; return r; }
    // partial sums of the CG's dot products and of k_cg_refine, each in slots of its own
    enum { kPartRz = 4, kPartPap, kPartRr, kPartRefine };
    static double *part(Instance &I, int slot) { return I.partials + (size_t)slot * I.red_stride; }


    // --- transport (Eq. alphaExp) ------------------------------------------
    template <int DIM>
    static int transport_d(Instance &I, void *const *phi, double dt) {
        GridD g = to_dev(I.g);
        L3 L = launch3(I.g);
        T rV = (T)(dt / I.g.V);
        launchk(k_transport_low<DIM, T>, L.grid, L.block, 0, I.stream, g, I.info, tp(I.alpha), c3(phi), c3(I.nf),
                                                                  (T)I.P.c_alpha, (T)I.P.alpha_inlet, rV, tp(I.aL),
                                                                  tp(I.Pp), tp(I.Pm)), ++I.nlaunch;
        launchk(k_transport_ratio<DIM, T>, L.grid, L.block, 0, I.stream, g, I.info, tp(I.alpha), tp(I.aL), tp(I.Pp),
                                                                    tp(I.Pm), rV, (T)(I.g.V / dt), tp(I.Rp), tp(I.Rm)), ++I.nlaunch;
        launchk(k_transport_update<DIM, T>, L.grid, L.block, 0, I.stream, g, I.info, tp(I.alpha), c3(phi), c3(I.nf),
                                                                     (T)I.P.c_alpha, tp(I.aL), tp(I.Rp), tp(I.Rm), rV,
                                                                     tp(I.alpha_new)), ++I.nlaunch;
        OSCAR_LAUNCH_CHECK();
        return 0;
    }
    static int transport(Instance &I, void *const *phi, double dt) {
        return I.g.dim == 3 ? transport_d<3>(I, phi, dt) : transport_d<2>(I, phi, dt);
    }

    // --- interface (Section 2.1) -------------------------------------------
    template <int DIM>
    static int interface_d(Instance &I, void *alpha) {
        GridD g = to_dev(I.g);
        L3 L = launch3(I.g);
        const GR<T> gr = to_gr<T>(I.g, 1.0);
        void *src = alpha;
        for (int pass = 0; pass < I.P.n_smooth; ++pass) {
            void *dst = (pass % 2 == 0) ? I.alpha_s : I.alpha_tmp;
            launchk(k_smooth<DIM, T>, L.grid, L.block, 0, I.stream, g, gr, I.info, tp(src), tp(dst)), ++I.nlaunch;
            src = dst;
        }
        const T *as = tp(src);
        T ct = (T)I.cos_theta, dn = (T)I.deltaN;
        L3 F0 = launch3_faces(I.g, 0), F1 = launch3_faces(I.g, 1), F2 = launch3_faces(I.g, 2);
        launchk(k_normals<DIM, 0, T>, F0.grid, F0.block, 0, I.stream, g, gr, I.info, as, ct, dn, tp(I.nf[0])), ++I.nlaunch;
        launchk(k_normals<DIM, 1, T>, F1.grid, F1.block, 0, I.stream, g, gr, I.info, as, ct, dn, tp(I.nf[1])), ++I.nlaunch;
        if (DIM == 3)
            launchk(k_normals<DIM, 2, T>, F2.grid, F2.block, 0, I.stream, g, gr, I.info, as, ct, dn, tp(I.nf[2])), ++I.nlaunch;
        launchk(k_curvature<DIM, T>, L.grid, L.block, 0, I.stream, g, gr, I.info, c3(I.nf), tp(I.kappa)), ++I.nlaunch;
        OSCAR_LAUNCH_CHECK();
        return 0;
    }
    static int interface_(Instance &I, void *alpha) {
        return I.g.dim == 3 ? interface_d<3>(I, alpha) : interface_d<2>(I, alpha);
    }

    // --- multigrid -----------------------------------------------------------
    static MG3<M> mg3(const Level &L) { MG3<M> c; for (int a = 0; a < 3; ++a) c.a[a] = (const M *)L.c[a]; return c; }

    // operators of every level and the coarsest one's inverse, on stream st
    template <int DIM>
    static int mg_coeffs_d(Instance &I, cudaStream_t st) {
        for (int l = 0; l < I.nlev; ++l) {
            Level &L = I.lev[l];
            GridD g = to_dev(L.g);
            L3 LL = launch3(L.g);
            if (l == 0) {
                launchx(false, 1, k_mg_diag<DIM, M>, LL.grid, LL.block, 0, st, g, L.fluid, mg3(L), (M *)L.diag,
                        (M *)L.idiag), ++I.nlaunch;
            } else {
                Level &F = I.lev[l - 1];
                P3<M> cc;
                for (int a = 0; a < 3; ++a) cc.a[a] = (M *)L.c[a];
                launchk(k_mg_level_operator<DIM, M>, LL.grid, LL.block, 0, st, to_dev(F.g), g, F.r[0], F.r[1],
                        F.r[2], mg3(F), cc, (const uint8_t *)L.fluid, (M *)L.diag, (M *)L.idiag), ++I.nlaunch;
            }
        }
        const Level &E = I.lev[exact_level(I, top_level(I))];
        if constexpr (sizeof(M) == sizeof(float))
            launchk(k_mg_inverse_dense<DIM>, 1, kGjThreads, 0, st, to_dev(E.g), mg3(E), (const M *)E.diag,
                    (const uint8_t *)E.fluid, (M *)I.cl_inv, I.coarse_refresh, (const int *)I.ctl), ++I.nlaunch;
        else
            launchk(k_mg_inverse_band<DIM, M>, (E.g.ncell + kBandCols - 1) / kBandCols, 32, inverse_smem(E.g), st, to_dev(E.g), mg3(E),
                    (const M *)E.diag, (const uint8_t *)E.fluid, (M *)I.cl_inv, I.coarse_refresh, (const int *)I.ctl),
                ++I.nlaunch;
        {   // the images of the levels the solves work in a cluster
            ClLevels<M> P;
            ClSolve A;
            if (I.solve_nc) cl_fill(I, P, 0, I.solve_nc, &A);
            else cl_fill(I, P, top_level(I), I.cl_nc);
            launchk(k_cl_pack<DIM, M>, dim3(P.nc, kPackSlices), kPackThreads, 0, st, P, I.ctl), ++I.nlaunch;
        }
        OSCAR_LAUNCH_CHECK();
        return 0;
    }

    // --- the cluster's levels ------------------------------------------------
    // first level worked by the V-cycle's cluster
    static int top_level(const Instance &I) { return I.lg >= 0 ? I.lg : I.lc0; }
    // the level solved with its explicit inverse below level l0
    static int exact_level(const Instance &I, int l0) {
        int l = l0;
        while (l < I.nlev - 1 && I.lev[l].g.ncell > kExactCells) ++l;
        return l;
    }
    static size_t inverse_smem(const GridH &g) {
        int e[3] = {g.nx, g.ny, g.nz};
        std::sort(e, e + 3);
        return band_words(band_shape(g.ncell, e[0] * e[1])) * sizeof(M);
    }

    // Levels l0 .. of a cluster of at most nc_max CTAs and their shared-memory
    // layout; returns the bytes each CTA needs, (size_t)-1 when the levels
    // cannot be worked by a cluster. With A the vectors of a whole solve are
    // laid out too.
    static size_t cl_fill(const Instance &I, ClLevels<M> &P, int l0, int nc_max, ClSolve *A = nullptr) {
        memset(&P, 0, sizeof(P));
        const int le = exact_level(I, A ? top_level(I) : l0);   // one inverse serves both kernels
        P.n = le - l0 + 1;
        if (P.n > kMaxCL || I.lev[le].g.ncell > kExactCells) return (size_t)-1;
        P.cols = I.lev[le].g.nx;
        P.nc = 1;
        while (2 * P.nc <= nc_max && 2 * P.nc <= P.cols) { P.nc *= 2; ++P.lnc; }
        P.inv = (const M *)I.cl_inv;
        size_t off = 0, rs = 0;
        auto take = [&](size_t bytes) { size_t o = off; off = (off + bytes + 15) & ~(size_t)15; return (int)o; };
        int w[kMaxCL], sh = 0;
        for (int q = P.n - 1; q >= 0; --q) {   // slabs, from the coarsest level
            const Level &L = I.lev[l0 + q];
            if (q < P.n - 1 && L.r[0] == 2) ++sh;
            P.L[q].sh = sh;
            w[q] = 0;
            for (int r = 0; r < P.nc; ++r) {
                const int s0 = std::min(((r * P.cols) >> P.lnc) << sh, L.g.nx);
                const int s1 = std::min((((r + 1) * P.cols) >> P.lnc) << sh, L.g.nx);
                w[q] = std::max(w[q], s1 - s0);
            }
        }
        int E = A ? 1 : 0;   // a solve applies the operator to z
        for (int q = 0; q < P.n; ++q) {
            const Level &L = I.lev[l0 + q];
            ClLevel<M> &C = P.L[q];
            const bool last = q == P.n - 1;
            C.nx = L.g.nx; C.ny = L.g.ny; C.nz = L.g.nz;
            C.rx = L.r[0]; C.ry = L.r[1]; C.rz = L.r[2];
            C.paired = l0 + q >= I.lc0;
            C.nu = l0 + q == 0 ? I.mg_nu : (l0 + q < I.lc0 ? I.mg_nu_c : I.mg_nu_cta);
            C.E = E;
            C.D = last ? E : E + 4 * C.nu - 2;
            // the ghosts held: at most the whole domain, at least the column beyond it
            C.G = P.nc == 1 ? 1 : std::min(C.nx, std::max(1, C.D));
            E = (E + 2 * C.nu + C.rx - 1) / C.rx;
            C.ncol = w[q] + 2 * C.G;
            C.ps = (C.ny * C.nz) | 1;
            const size_t n = (size_t)C.ncol * C.ps;
            if (n > 65534) return (size_t)-1;   // list entries hold 16-bit cell numbers
            C.nloc = (int)n;
            C.ce = ((C.ny + 1) / 2) * C.nz;
            C.rncol = 1.0f / (float)C.ncol;
            C.rny = 1.0f / (float)C.ny;
            C.rce = 1.0f / (float)C.ce;
            for (int a = 0; a < 3; ++a) C.c[a] = (const M *)L.c[a];
            C.idiag = (const M *)L.idiag;
            C.oi = take(n * sizeof(M));
            for (int a = 0; a < L.g.dim; ++a) C.oc[a] = take(n * sizeof(M));
            const size_t nh = (size_t)C.ncol * C.ce * sizeof(unsigned short);
            C.ol[0] = take(nh);
            C.ol[1] = take(nh);
            if (!last) C.op = take(nh);
            C.os = take((P.nc + 1) * sizeof(short));
            if (C.nx > 32767) return (size_t)-1;   // slab starts are 16-bit numbers
            if (!last) rs = std::max(rs, (size_t)w[q] * C.ps);
        }
        const ClLevel<M> &Lc = P.L[P.n - 1];
        const size_t ne = I.lev[le].g.ncell;
        const size_t nrow = std::min((size_t)(w[P.n - 1] + 2 * cl_exact_depth(P)) * Lc.ny * Lc.nz, ne);
        P.oinv = take(nrow * ne * sizeof(M));
        P.orow = take(nrow * sizeof(unsigned short));
        P.img = (int)off;
        P.image = (unsigned char *)I.cl_image;
        for (int q = 0; q < P.n; ++q) {
            P.L[q].ox = take((size_t)P.L[q].nloc * sizeof(M));
            P.L[q].ob = take((size_t)P.L[q].nloc * sizeof(M));
        }
        if (A) rs = std::max(rs, (size_t)w[0] * P.L[0].ps);   // the products of a dot
        P.ors = take(rs * sizeof(M));
        P.obx = take(ne * sizeof(M));
        if (A) {
            P.ored = take((4 * solve_threads(I.g.ncell) + 2 * 4 * kMaxCluster) * sizeof(double));
            const size_t n = (size_t)(w[0] + 2) * P.L[0].ps;
            A->op = take(n * sizeof(M));
            A->oap = take(n * sizeof(M));
            A->oe = sizeof(M) == sizeof(float) ? take(n * sizeof(M)) : A->oap;
        }
        return off;
    }

    // rows of the first level that a CTA with the widest slab works
    static long long cl_rows(const ClLevels<M> &P) {
        const ClLevel<M> &L = P.L[0];
        return (long long)std::min(L.nx, L.ncol - 2 * L.G + 2 * std::min(L.D, L.nx)) * L.ny * L.nz;
    }

    // x / b of level l (level 0 works in place on the Krylov vectors z / r)
    static M *lx(Instance &I, int l, V *z) { return l == 0 ? (M *)z : (M *)I.lev[l].x; }
    static M *lb(Instance &I, int l, V *r) { return l == 0 ? (M *)r : (M *)I.lev[l].b; }

    // FP32 levels whose half sweeps stream from HBM (the coefficients, x, b and
    // the inverse diagonal beyond what L2 keeps beside the other vectors) form
    // the inverse diagonal instead of reading it. Whole steps without and with
    // it: 256x128x128 (101 MB) 24.08 and 23.60 ms; 208x104x104 (54 MB) 14.78 and
    // 15.11, 2048x1024 (42 MB) 21.73 and 22.00.
    static constexpr double kStreamBytes = 80e6;
    static bool diag_from_rows(const GridH &g) {
        return sizeof(M) == sizeof(float) && (g.dim + 3.0) * g.ncell * sizeof(M) >= kStreamBytes;
    }
    // one half sweep; with_dot (finest level only) also forms r.z and beta
    template <int DIM>
    static void smooth_level(Instance &I, int l, int colour, M *x, const M *b, bool with_dot = false) {
        Level &L = I.lev[l];
        GridD g = to_dev(L.g);
        L3 LL = launch3((L.g.nx + 1) / 2, L.g.ny, L.g.nz);
        if (with_dot) {
            const L3G LD = launch_groups((L.g.nx + 1) / 2, L.g.ny * L.g.nz, kDotRows<M>);
            launchk(k_mg_rbgs_dot<DIM, M, kDotRows<M>>, LD.grid, LD.block, 0, I.stream, g, mg3(L), (const M *)L.idiag, x, b, colour,
                    LD.groups, part(I, kPartRz)), ++I.nlaunch;
            I.nrz = LD.nblocks;
        } else
            for (int rep = 0; rep < (l == 0 && I.repeat_fine ? 2 : 1); ++rep)   // a repeat is idempotent
                launchk(diag_from_rows(L.g) ? k_mg_rbgs<DIM, M, false, sizeof(M) == sizeof(float)> : k_mg_rbgs<DIM, M, false, false>,
                        LL.grid, LL.block, 0, I.stream, g, mg3(L), (const M *)L.idiag, x, b, colour, g, 0, 0, 0,
                        (const M *)nullptr), ++I.nlaunch;
    }
    // the first post-smoothing half sweep (colour 1) of level l with the
    // prolongation from level l + 1 (x of level l + 1 in xc) folded in
    template <int DIM>
    static void prolong_smooth(Instance &I, int l, M *x, const M *b, const M *xc) {
        Level &L = I.lev[l], &C = I.lev[l + 1];
        GridD g = to_dev(L.g), gc = to_dev(C.g);
        L3 LL = launch3((L.g.nx + 1) / 2, L.g.ny, L.g.nz);
        launchk(diag_from_rows(L.g) ? k_mg_rbgs<DIM, M, true, sizeof(M) == sizeof(float)> : k_mg_rbgs<DIM, M, true, false>, LL.grid, LL.block, 0, I.stream, g, mg3(L), (const M *)L.idiag, x, b, 1, gc,
                L.r[0] >> 1, L.r[1] >> 1, L.r[2] >> 1, xc), ++I.nlaunch;
    }

    template <int DIM, int RX, int RY, int RZ>
    static void rr_launch(Instance &I, const Level &L, const Level &C, const M *x, const M *b, M *bc, M *xc, int first) {
        using TT = RRTile<DIM>;
        const dim3 grid((L.g.nx + TT::X - 1) / TT::X, (L.g.ny + TT::Y - 1) / TT::Y, (L.g.nz + TT::Z - 1) / TT::Z);
        launchk(k_mg_resid_restrict<DIM, M, RX, RY, RZ>, grid, dim3(TT::X, TT::Y, TT::Z), 0, I.stream, to_dev(L.g),
                to_dev(C.g), mg3(L), (const M *)L.diag, x, b, bc, xc, (const M *)C.idiag, first);
        ++I.nlaunch;
    }
    // fused residual + restriction (+ the coarse level's first colour-0 half
    // sweep when first is set), dispatched on the coarsening ratios
    template <int DIM>
    static void resid_restrict(Instance &I, const Level &L, const Level &C, const M *x, const M *b, M *bc, M *xc,
                               int first) {
        int code = (L.r[0] == 2) | ((L.r[1] == 2) << 1) | ((L.r[2] == 2) << 2);
        switch (code) {
            case 1: rr_launch<DIM, 2, 1, 1>(I, L, C, x, b, bc, xc, first); break;
            case 2: rr_launch<DIM, 1, 2, 1>(I, L, C, x, b, bc, xc, first); break;
            case 3: rr_launch<DIM, 2, 2, 1>(I, L, C, x, b, bc, xc, first); break;
            case 4: rr_launch<DIM, 1, 1, 2>(I, L, C, x, b, bc, xc, first); break;
            case 5: rr_launch<DIM, 2, 1, 2>(I, L, C, x, b, bc, xc, first); break;
            case 6: rr_launch<DIM, 1, 2, 2>(I, L, C, x, b, bc, xc, first); break;
            case 7: rr_launch<DIM, 2, 2, 2>(I, L, C, x, b, bc, xc, first); break;
            default: rr_launch<DIM, 1, 1, 1>(I, L, C, x, b, bc, xc, first); break;
        }
    }

    // z = V-cycle(r): pre-smoothing red-black, post-smoothing black-red
    // (symmetric, so a valid CG preconditioner); levels from top_level down run
    // in one cluster. The first colour-0 half sweep of each level above it is
    // done by the kernel that produces its right-hand side (k_cg_init /
    // k_cg_update for the finest level, the restriction for the others).
    template <int DIM>
    static int vcycle_d(Instance &I, V *r, V *z) {
        const int lk = top_level(I);   // first level not worked by per-level kernels
        for (int l = 0; l < lk; ++l) {
            Level &L = I.lev[l], &C = I.lev[l + 1];
            M *x = lx(I, l, z), *b = lb(I, l, r);
            int nu = l == 0 ? I.mg_nu : I.mg_nu_c;
            for (int s = 0; s < nu; ++s) {
                if (s > 0) smooth_level<DIM>(I, l, 0, x, b);
                smooth_level<DIM>(I, l, 1, x, b);
            }
            resid_restrict<DIM>(I, L, C, x, b, lb(I, l + 1, r), lx(I, l + 1, z), l + 1 < lk ? 1 : 0);
        }
        {
            ClLevels<M> P;
            cl_fill(I, P, lk, I.cl_nc);
            launchx(true, P.nc, k_mg_cluster<DIM, M>, P.nc, kVcycleThreads, I.cl_smem, I.stream, P,
                    (const M *)lb(I, lk, r), lx(I, lk, z)), ++I.nlaunch;
        }
        for (int l = lk - 1; l >= 0; --l) {
            M *x = lx(I, l, z), *b = lb(I, l, r);
            int nu = l == 0 ? I.mg_nu : I.mg_nu_c;
            for (int s = 0; s < nu; ++s) {
                if (s == 0) prolong_smooth<DIM>(I, l, x, b, (const M *)lx(I, l + 1, z));
                else smooth_level<DIM>(I, l, 1, x, b);
                smooth_level<DIM>(I, l, 0, x, b, l == 0 && s == nu - 1);   // the last one also forms r.z
            }
        }
        OSCAR_LAUNCH_CHECK();
        return 0;
    }

    // r = b - M q (FP64), ||b||^2, ||r||^2 into S_BB, S_RR, then the loop
    // decision of residual_control(mode)
    // (with_E: also the normalised residual E_k of Section 3.2 for q, b)
    template <int DIM>
    static void residual64(Instance &I, const double *q, const double *b, int mode, cudaGraphConditionalHandle h,
                           V *zero1, V *zero2, double *r64 = nullptr, bool with_E = false) {
        GridD g = to_dev(I.g);
        L3 L = launch_rows(I.g, kRedBlocks);
        launchk(k_cg_init<DIM, T, V>, L.grid, L.block, 0, I.stream, g, I.info, w64(I), q, b, (V *)I.cg_r, r64,
                (const V *)I.lev[0].idiag, (V *)I.cg_z, zero1, zero2, I.partials, I.red_stride, I.ticket, L.nblocks,
                I.scal, I.ctl, I.P.cg_rtol, mode, h, with_E ? 1.0 / (double)I.n_fluid : 0.0), ++I.nlaunch;
    }

    // one PCG iteration on M x = r with Krylov vectors z, p, Ap (type V), up to
    // the update; nrr: partials of r.r left in kPartRr
    template <int DIM>
    static int pcg_body(Instance &I, V *x, int xfresh, int *nrr) {
        GridD g = to_dev(I.g);
        const int n = I.g.ncell, rows = I.g.ny * I.g.nz;
        V *r = (V *)I.cg_r, *z = (V *)I.cg_z, *p = (V *)I.cg_p, *Ap = (V *)I.cg_Ap;
        OSCAR_TRY(vcycle_d<DIM>(I, r, z));
        if (top_level(I) == 0) {   // the whole V-cycle ran in the cluster: r.z on its own
            I.nrz = std::min(kDotBlocks, nblk(n));
            launchk(k_cg_dot_rz<V>, I.nrz, BS, 0, I.stream, n, r, z, part(I, kPartRz)), ++I.nlaunch;
        }
        int npap;
        if constexpr (sizeof(V) == sizeof(float)) {
            const L3G LA = launch_groups(I.g.nx, rows, kApplyRows);
            npap = LA.nblocks;
            launchk(k_cg_pz_apply<DIM, T, V, kApplyRows>, LA.grid, LA.block, 0, I.stream, g, c3(I.lev[0].c),
                    (const V *)z, p, Ap, part(I, kPartRz), I.nrz, part(I, kPartPap), LA.groups, I.scal, I.ctl), ++I.nlaunch;
        } else {   // FP64 path: the search direction as written, M p applied directly
            launchk(k_cg_pupdate<V>, std::min(kDotBlocks, nblk(n)), BS, 0, I.stream, n, (const V *)z, p,
                    part(I, kPartRz), I.nrz, I.scal, I.ctl), ++I.nlaunch;
            const L3G LA = launch_groups(I.g.nx, rows, 1);
            npap = LA.nblocks;
            launchk(k_cg_apply_dot<DIM, V>, LA.grid, LA.block, 0, I.stream, g, c3(I.lev[0].c), (const V *)p, Ap,
                    part(I, kPartPap), LA.groups), ++I.nlaunch;
        }
        const L3G LU = launch_groups(I.g.nx, rows, kUpdateRows);
        launchk(k_cg_update<V, kUpdateRows>, LU.grid, LU.block, 0, I.stream, g, x, r, p, Ap, (const V *)I.lev[0].idiag,
                z, part(I, kPartPap), npap, part(I, kPartRr), LU.groups, I.scal, (const int *)I.ctl, xfresh), ++I.nlaunch;
        *nrr = LU.nblocks;
        OSCAR_LAUNCH_CHECK();
        return 0;
    }

    // Pressure solve M q = b. FP64 path: PCG on q itself. Mixed path: FP64
    // defect correction around an FP32 PCG for the correction e, as one loop of
    // PCG iterations (k_cg_refine ends a trip).
    template <int DIM>
    static int pcg_d(Instance &I, double *q, const double *b, bool with_E) {
        if (DIM == 2 && I.solve_nc) {
            ClLevels<M> P;
            ClSolve A;
            memset(&A, 0, sizeof(A));
            cl_fill(I, P, 0, I.solve_nc, &A);
            A.g = to_dev(I.g);
            A.info = I.info;
            A.w64 = w64(I);
            A.q = q;
            A.b = b;
            A.r64 = I.cg_r64;
            A.scal = I.scal;
            A.ctl = I.ctl;
            A.rtol = I.P.cg_rtol;
            A.inv_nf = with_E ? 1.0 / (double)I.n_fluid : 0.0;
            A.maxit = I.P.cg_maxit;
            A.by = (int)launch3(I.g).block.y;
            launchx(!with_E, P.nc, k_solve_cluster<T>, P.nc, solve_threads(I.g.ncell), I.solve_smem, I.stream, P, A), ++I.nlaunch;
            OSCAR_LAUNCH_CHECK();
            return 0;
        }
        constexpr bool mixed = sizeof(T) == sizeof(float);
        cudaGraphConditionalHandle h;
        OSCAR_TRY(cond_handle(I, &h));
        // mixed: the iteration starts e and p from 0 itself (xfresh, beta = 0),
        // so neither is cleared; the FP64 residual is evaluated once, then
        // updated by k_cg_refine at the end of every trip
        residual64<DIM>(I, q, b, mixed ? 1 : 0, h, mixed ? nullptr : (V *)I.cg_p, nullptr, mixed ? I.cg_r64 : nullptr, with_E);
        return loop_while(I, h, [&]() -> int {
            const long long n0 = I.nlaunch;
            int nrr = 0;
            OSCAR_TRY(pcg_body<DIM>(I, mixed ? (V *)I.cg_e : (V *)q, mixed ? 1 : 0, &nrr));
            if constexpr (mixed) {
                const L3 L = launch_sms(I.g);
                launchk(k_cg_refine<DIM>, L.grid, L.block, 0, I.stream, to_dev(I.g), I.info, c3(I.lev[0].c),
                        (const float *)I.cg_e, q, I.cg_r64, (float *)I.cg_r, (const float *)I.lev[0].idiag,
                        (float *)I.cg_z, part(I, kPartRr), nrr, part(I, kPartRefine), I.red_stride, I.ticket, L.nblocks,
                        I.scal, I.ctl, I.P.cg_rtol, I.P.cg_maxit, h), ++I.nlaunch;
            } else {
                launchk(k_cg_check<V>, 1, BS, 0, I.stream, part(I, kPartRr), nrr, I.scal, I.ctl, I.P.cg_maxit, h),
                    ++I.nlaunch;
            }
            if (I.capturing) {
                I.n_cg_body = I.nlaunch - n0;
                I.cg_bodies_captured += 1;
            }
            OSCAR_LAUNCH_CHECK();
            return 0;
        });
    }

    // --- PISO (Section 2.2) --------------------------------------------------
    template <int DIM>
    static int piso_d(Instance &I, void *const *v, double *q, void *const *phi, bool has_st, double vin0, double dt) {
        GridD g = to_dev(I.g);
        L3 L = launch3(I.g);
        L3 F[3] = {launch3_faces(I.g, 0), launch3_faces(I.g, 1), launch3_faces(I.g, 2)};
        const GR<T> gr = to_gr<T>(I.g, dt);
        Fluid<T> fl{(T)I.P.rho1, (T)I.P.rho2, (T)I.P.mu1, (T)I.P.mu2};
        const T *al = tp(I.alpha_new);
        launchk(k_rA<DIM, T>, L.grid, L.block, 0, I.stream, g, gr, I.info, al, c3(I.phic), fl, (T)dt, tp(I.rA)), ++I.nlaunch;
        void **cf = I.lev[0].c;
        T sig = (T)I.P.sigma;
        int st = has_st ? 1 : 0;
        launchk(k_face_coeffs<0, T>, F[0].grid, F[0].block, 0, I.stream, g, gr, I.info, tp(I.rA), tp(I.kappa), al, sig, st,
                                                                    tp(cf[0]), tp(I.fst[0]), cf64_out(I, 0)), ++I.nlaunch;
        launchk(k_face_coeffs<1, T>, F[1].grid, F[1].block, 0, I.stream, g, gr, I.info, tp(I.rA), tp(I.kappa), al, sig, st,
                                                                    tp(cf[1]), tp(I.fst[1]), cf64_out(I, 1)), ++I.nlaunch;
        if (DIM == 3)
            launchk(k_face_coeffs<2, T>, F[2].grid, F[2].block, 0, I.stream, g, gr, I.info, tp(I.rA), tp(I.kappa), al, sig, st,
                                                                        tp(cf[2]), tp(I.fst[2]), cf64_out(I, 2)), ++I.nlaunch;
        OSCAR_LAUNCH_CHECK();
        // the multigrid operators are first needed by the solve: they are built
        // on a branch beside the first momentum prediction. A timed step keeps
        // them on the instance's stream: no kernel is timed beside another, and the
        // recording waits for that stream only
        const bool branch = !t_prof;
        if (branch && (cudaEventRecord(I.ev_fork, I.stream) != cudaSuccess ||
                       cudaStreamWaitEvent(I.aux, I.ev_fork, 0) != cudaSuccess))
            return OSCAR_E_CUDA;
        OSCAR_TRY(mg_coeffs_d<DIM>(I, branch ? I.aux : I.stream));
        if (branch && cudaEventRecord(I.ev_join, I.aux) != cudaSuccess) return OSCAR_E_CUDA;
        P3<T> Gp0 = p3(&I.G[0]), Gp1 = p3(&I.G[3]), Gp2 = p3(&I.G[6]);
        C3<T> Gc0 = c3(&I.G[0]), Gc1 = c3(&I.G[3]), Gc2 = c3(&I.G[6]);
        for (int corr = 0; corr < I.P.n_piso; ++corr) {
            launchk(k_vel_grad<DIM, T>, L.grid, L.block, 0, I.stream, g, gr, I.info, c3(v), (T)vin0, Gp0, Gp1, Gp2), ++I.nlaunch;
            launchk(k_momentum_H<DIM, T>, L.grid, L.block, 0, I.stream, g, gr, I.info, c3(v), c3(I.vold), c3(I.phic), al,
                                                                   tp(I.rA), fl, (T)vin0, (T)dt, Gc0, Gc1, Gc2,
                                                                   p3(I.hbya)), ++I.nlaunch;
            launchk(k_phistar_rhs<DIM, T>, L.grid, L.block, 0, I.stream, g, I.info, c3(I.hbya), tp(I.rA), c3(I.fst),
                    (T)vin0, p3(I.phis), I.cg_b), ++I.nlaunch;
            // E_k, the normalised initial residual of the first corrector
            // (Section 3.2), is formed by the solve's initial-residual kernel
            if (corr == 0) {
                if (branch && cudaStreamWaitEvent(I.stream, I.ev_join, 0) != cudaSuccess) return OSCAR_E_CUDA;
                if (!(DIM == 2 && I.solve_nc))   // the one-launch solve sums q itself
                    launchx(false, 1, k_sum_to<double>, kRedBlocks, BS, 0, I.stream, g.ncell, q, 1.0, I.partials,
                            I.ticket, I.scal, S_QSUM), ++I.nlaunch;
            }
            OSCAR_LAUNCH_CHECK();
            OSCAR_TRY(pcg_d<DIM>(I, q, I.cg_b, corr == 0));
            launchk(k_correct<DIM, T>, L.grid, L.block, 0, I.stream, g, gr, I.info, c3(I.phis), c3(cf), q, p3(phi),
                    c3(I.hbya), tp(I.rA), c3(I.fst), p3(v)), ++I.nlaunch;
            OSCAR_LAUNCH_CHECK();
        }
        return 0;
    }
    static int piso(Instance &I, void *const *v, double *q, void *const *phi, bool has_st, double vin0, double dt) {
        return I.g.dim == 3 ? piso_d<3>(I, v, q, phi, has_st, vin0, dt) : piso_d<2>(I, v, q, phi, has_st, vin0, dt);
    }

    static int copy_fields(Instance &I, void *const *dst, void *const *src, int is_face) {
        for (int a = 0; a < I.g.dim; ++a) {
            size_t n = is_face ? I.g.nf[a] : I.g.ncell;
            if (cudaMemcpyAsync(dst[a], src[a], n * sizeof(T), cudaMemcpyDeviceToDevice, I.stream) != cudaSuccess)
                return OSCAR_E_CUDA;
        }
        return 0;
    }
    static int sum_faces(Instance &I, void *const *a, void *const *b, void *const *out) {
        for (int d = 0; d < I.g.dim; ++d)
            launchk(k_sum2<T>, nblk(I.g.nf[d]), BS, 0, I.stream, I.g.nf[d], tp(a[d]), tp(b[d]), tp(out[d])), ++I.nlaunch;
        OSCAR_LAUNCH_CHECK();
        return 0;
    }
    // scal[slot] = sigma A + kinetic energy of u_cr (the energy exit test)
    static int relax_energy(Instance &I, int slot) {
        GridD g = to_dev(I.g);
        Fluid<T> fl{(T)I.P.rho1, (T)I.P.rho2, (T)I.P.mu1, (T)I.P.mu2};
        if (I.g.dim == 3)
            launchk(k_relax_energy<3, T>, kRedBlocks, BS, 0, I.stream, I.g.ncell, g, to_gr<T>(I.g, 1.0), I.info, (const T *)I.alpha,
                    c3(I.u_cr), fl, I.P.sigma, I.partials, I.red_stride, I.ticket, I.scal, slot), ++I.nlaunch;
        else
            launchk(k_relax_energy<2, T>, kRedBlocks, BS, 0, I.stream, I.g.ncell, g, to_gr<T>(I.g, 1.0), I.info, (const T *)I.alpha,
                    c3(I.u_cr), fl, I.P.sigma, I.partials, I.red_stride, I.ticket, I.scal, slot), ++I.nlaunch;
        OSCAR_LAUNCH_CHECK();
        return 0;
    }
    static int commit_alpha(Instance &I) {
        return cudaMemcpyAsync(I.alpha, I.alpha_new, (size_t)I.g.ncell * sizeof(T), cudaMemcpyDeviceToDevice,
                               I.stream) == cudaSuccess ? 0 : OSCAR_E_CUDA;
    }
    static int load_ctl(Instance &I) {
        return cudaMemcpyAsync(I.ctl, I.ctl_host, C_COUNT * sizeof(int), cudaMemcpyHostToDevice, I.stream) ==
                       cudaSuccess ? 0 : OSCAR_E_CUDA;
    }

    // --- step bodies ---------------------------------------------------------
    // Section 3.1: viscous-drag step
    static int body_drag(Instance &I, double dt) {
        OSCAR_TRY(load_ctl(I));
        OSCAR_TRY(transport(I, I.phi_vd, dt));
        OSCAR_TRY(sum_faces(I, I.phi_vd, I.phi_cr, I.phic));
        OSCAR_TRY(copy_fields(I, I.vold, I.u_vd, 0));
        OSCAR_TRY(piso(I, I.u_vd, I.p_vd, I.phi_vd, false, I.P.U_inlet, dt));
        OSCAR_TRY(commit_alpha(I));
        return interface_(I, I.alpha);
    }
    // Section 2.2: standard time-stepping
    static int body_standard(Instance &I, double dt) {
        OSCAR_TRY(load_ctl(I));
        OSCAR_TRY(transport(I, I.phi_vd, dt));
        OSCAR_TRY(interface_(I, I.alpha_new));
        OSCAR_TRY(copy_fields(I, I.phic, I.phi_vd, 1));
        OSCAR_TRY(copy_fields(I, I.vold, I.u_vd, 0));
        OSCAR_TRY(piso(I, I.u_vd, I.p_vd, I.phi_vd, true, I.P.U_inlet, dt));
        OSCAR_TRY(commit_alpha(I));
        for (int a = 0; a < I.g.dim; ++a)
            if (cudaMemsetAsync(I.u_sum[a], 0, I.g.ncell * sizeof(double), I.stream) != cudaSuccess)
                return OSCAR_E_CUDA;
        return 0;
    }
    // Section 3.2: relaxation loop with the early exit on the device
    static int body_relax(Instance &I, double dt, long long *n_pre, long long *n_body) {
        long long s0 = I.nlaunch;
        OSCAR_TRY(load_ctl(I));
        for (int a = 0; a < I.g.dim; ++a)
            if (cudaMemsetAsync(I.u_sum[a], 0, I.g.ncell * sizeof(double), I.stream) != cudaSuccess)
                return OSCAR_E_CUDA;
        cudaGraphConditionalHandle h;
        OSCAR_TRY(cond_handle(I, &h));
        const bool area = I.P.conv_mode == OSCAR_CONV_AREA;
        if (area) OSCAR_TRY(relax_energy(I, S_AREA0));
        launchk(k_relax_init, 1, 1, 0, I.stream, I.ctl, h), ++I.nlaunch;
        *n_pre = I.nlaunch - s0;
        long long b0 = I.nlaunch, cg0 = I.cg_bodies_captured;
        int rc = loop_while(I, h, [&]() -> int {
            OSCAR_TRY(transport(I, I.phi_cr, dt));
            OSCAR_TRY(interface_(I, I.alpha_new));
            OSCAR_TRY(sum_faces(I, I.phi_vd, I.phi_cr, I.phic));
            OSCAR_TRY(copy_fields(I, I.vold, I.u_cr, 0));
            OSCAR_TRY(piso(I, I.u_cr, I.p_cr, I.phi_cr, true, 0.0, dt));
            OSCAR_TRY(commit_alpha(I));
            if (area) OSCAR_TRY(relax_energy(I, S_AREA1));
            P3<double> us;
            for (int a = 0; a < 3; ++a) us.a[a] = I.u_sum[a];
            double invU = I.P.U_inlet > 0 ? 1.0 / I.P.U_inlet : 0.0;
            if (I.g.dim == 3)
                launchk(k_relax_accum<3, T>, kRedBlocks, BS, 0, I.stream, I.g.ncell, I.info, c3(I.u_cr), c3(I.vold), us,
                                                                     I.partials, I.ticket, I.scal, I.ctl,
                                                                     I.P.conv_mode, I.P.conv_tol, invU, h), ++I.nlaunch;
            else
                launchk(k_relax_accum<2, T>, kRedBlocks, BS, 0, I.stream, I.g.ncell, I.info, c3(I.u_cr), c3(I.vold), us,
                                                                     I.partials, I.ticket, I.scal, I.ctl,
                                                                     I.P.conv_mode, I.P.conv_tol, invU, h), ++I.nlaunch;
            OSCAR_LAUNCH_CHECK();
            return 0;
        });
        // launches of one sub-step outside the loop bodies of its pressure solves
        *n_body = (I.nlaunch - b0) - (I.cg_bodies_captured - cg0) * I.n_cg_body;
        return rc;
    }

    static int build(Instance &I, int kind, double dt) {
        GraphSlot &G = I.gslot[kind];
        if (G.valid && G.dt == dt) return 0;
        if (G.valid) {
            cudaGraphExecDestroy(G.exec);
            cudaGraphDestroy(G.graph);
            G.valid = 0;
        }
        if (cudaStreamBeginCapture(I.stream, cudaStreamCaptureModeRelaxed) != cudaSuccess) return OSCAR_E_CUDA;
        I.capturing = 1;
        I.depth = 0;
        long long s0 = I.nlaunch, cg0 = I.cg_bodies_captured;
        long long n_pre = 0, n_body = 0;
        int rc;
        if (kind == 0) rc = body_drag(I, dt);
        else if (kind == 1) rc = body_relax(I, dt, &n_pre, &n_body);
        else rc = body_standard(I, dt);
        if (kind != 1) n_pre = (I.nlaunch - s0) - (I.cg_bodies_captured - cg0) * I.n_cg_body;
        cudaGraph_t graph = nullptr;
        cudaError_t e = cudaStreamEndCapture(I.stream, &graph);
        I.capturing = 0;
        if (rc || e != cudaSuccess) {
            if (graph) cudaGraphDestroy(graph);
            cudaGetLastError();
            return rc ? rc : OSCAR_E_CUDA;
        }
        if (cudaGraphInstantiate(&G.exec, graph, 0) != cudaSuccess) {
            cudaGraphDestroy(graph);
            cudaGetLastError();
            return OSCAR_E_CUDA;
        }
        G.graph = graph;
        G.dt = dt;
        G.valid = 1;
        G.n_pre = n_pre;
        G.n_body = n_body;
        return 0;
    }

    // Launch step `kind` (graph, or eager loops) and read its control words back.
    // launch one step (graph, or the eager sequence) and the copies of its
    // device scalars back to the host, without waiting
    static bool eager_now(const Instance &I) { return I.eager || (I.prof && I.prof->enabled); }
    static int run_launch(Instance &I, int kind, double dt, int N) {
        BlockXScope bxs(I.block_x);
        const bool eager = eager_now(I);
        if (!eager) OSCAR_TRY(build(I, kind, dt));
        OSCAR_TRY(sync_bounded(I.stream, kSyncTimeoutSec));   // ctl_host is read by the graph
        for (int q = 0; q < C_COUNT; ++q) I.ctl_host[q] = 0;
        I.ctl_host[C_N] = N;
        if (eager) {
            long long l0 = I.nlaunch, d0 = 0, d1 = 0;
            t_prof = (I.prof && I.prof->enabled) ? I.prof : nullptr;
            int rc = kind == 0 ? body_drag(I, dt) : kind == 1 ? body_relax(I, dt, &d0, &d1) : body_standard(I, dt);
            t_prof = nullptr;
            if (rc) return rc;
            I.nexec += I.nlaunch - l0;
        } else if (cudaGraphLaunch(I.gslot[kind].exec, I.stream) != cudaSuccess) {
            return OSCAR_E_CUDA;
        }
        if (cudaMemcpyAsync(I.scal_host, I.scal, S_COUNT * sizeof(double), cudaMemcpyDeviceToHost, I.stream) !=
                cudaSuccess ||
            cudaMemcpyAsync(I.ctl_host, I.ctl, C_COUNT * sizeof(int), cudaMemcpyDeviceToHost, I.stream) !=
                cudaSuccess)
            return OSCAR_E_CUDA;
        I.pending = kind;
        I.pending_dt = dt;
        I.pending_N = N;
        return 0;
    }
    static int run(Instance &I, int kind, double dt, int N) {
        OSCAR_TRY(run_launch(I, kind, dt, N));
        return run_finish(I);
    }
    // wait for the launched step and account for it
    static int run_finish(Instance &I) {
        const int kind = I.pending;
        const double dt = I.pending_dt;
        I.pending = -1;
        OSCAR_TRY(sync_bounded(I.stream, kSyncTimeoutSec));
        const GraphSlot &G = I.gslot[kind];
        int its = I.ctl_host[C_ITSUM];
        int trips = kind == 1 ? I.ctl_host[C_K] : 1;
        if (!eager_now(I)) {
            I.nexec += G.n_pre + (long long)(kind == 1 ? trips : 0) * G.n_body + (long long)its * I.n_cg_body;
        }
        I.cg_iters_last = its;
        I.cg_iters_total += its;
        I.cell_updates += (long long)trips * I.n_fluid;
        I.last_dt = dt;
        if (I.ctl_host[C_NAN]) return OSCAR_E_NAN;
        return I.ctl_host[C_NOTCONV] ? OSCAR_E_NOT_CONVERGED : 0;
    }
};

template <typename T> void Solver<T>::release_graphs(Instance &I) {
    I.n_cg_body = 0;   // set again by the next capture
    for (int k = 0; k < 3; ++k) {
        GraphSlot &G = I.gslot[k];
        if (G.valid) {
            cudaGraphExecDestroy(G.exec);
            cudaGraphDestroy(G.graph);
            G.valid = 0;
        }
    }
}

// The cluster takes the levels of at most `cap` cells whose subtree fits its
// shared memory; with cta_global it has several CTAs and takes the levels of
// at most vcycle_cells * cap cells and kVcycleRows per CTA (never the finest one,
// whose x and b are the Krylov vectors), and a small 2D grid's whole solve runs in one cluster.
template <typename T> int Solver<T>::choose_cta(Instance &I, long long cap) {
    ClLevels<T> P;
    const size_t budget = kClSmemBytes;
    if (cap > kCtaCells) cap = kCtaCells;
    const int nc = I.cta_global ? std::min(kVcycleCtas, I.cl_fit) : 1;
    const int keep = I.lc0;
    auto fits = [&](int l) { return Impl<T>::cl_fill(I, P, l, nc) <= budget; };
    int lc0 = I.nlev - 1;
    for (;;) {   // the layout depends on which levels take mg_nu_cta sweeps
        I.lc0 = lc0;
        if (!fits(lc0)) break;
        if (lc0 == 0 || I.lev[lc0 - 1].g.ncell > cap) { --lc0; break; }
        --lc0;
    }
    I.lc0 = ++lc0;   // the last one that fitted
    if (lc0 == I.nlev) { I.lc0 = keep; return OSCAR_E_INVALID_ARG; }
    int lg = lc0;
    if (I.cta_global)
        while (lg - 1 >= 1 && I.lev[lg - 1].g.ncell <= ClRule<T>::vcycle_cells * cap && fits(lg - 1) &&
               Impl<T>::cl_rows(P) <= kVcycleRows)
            --lg;
    I.lg = lg < lc0 ? lg : -1;
    I.cl_smem = Impl<T>::cl_fill(I, P, lg, nc);
    I.cl_nc = P.nc;
    I.cl_image_need = (size_t)P.img * P.nc;
    I.solve_nc = 0;
    if (I.cta_global && I.g.dim == 2 && I.g.ncell <= kSolveCells) {
        ClSolve A;
        I.solve_smem = Impl<T>::cl_fill(I, P, 0, std::min(solve_ctas<T>(I.g.ncell), I.solve_fit), &A);
        if (I.solve_smem <= budget && (P.nc == 1 || P.L[0].sh > 0)) {   // even slab starts
            I.solve_nc = P.nc;
            I.cl_image_need = (size_t)P.img * P.nc;
        }
    }
    return 0;
}

// The CTAs, at most nc, of a cluster of kernel f that the GPU can place. A GPU
// processing cluster with fewer SMs left than a cluster needs (16 CTAs of up to
// 220 KB take 16 SMs; a device with SMs turned off or partitioned) cannot hold
// it, and its launch would fail.
inline int cluster_fit(const void *f, int threads, int nc) {
    for (; nc > 1; nc /= 2) {
        cudaLaunchConfig_t cfg;
        memset(&cfg, 0, sizeof(cfg));
        cfg.gridDim = dim3(nc);
        cfg.blockDim = dim3(threads);
        cfg.dynamicSmemBytes = kClSmemBytes;
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = (unsigned)nc;
        attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, f, &cfg) == cudaSuccess && n > 0) break;
        cudaGetLastError();
    }
    return nc;
}

template <typename T> int Solver<T>::setup(Instance &I, const uint8_t *solid_dev, const double *alpha0_dev) {
    BlockXScope bxs(I.block_x);
    GridD g = to_dev(I.g);
    L3 L = launch3(I.g);
    long long l0 = I.nlaunch;
    if (I.g.dim == 3) launchk(k_build_info<3>, L.grid, L.block, 0, I.stream, g, solid_dev, I.info, I.lev[0].fluid), ++I.nlaunch;
    else launchk(k_build_info<2>, L.grid, L.block, 0, I.stream, g, solid_dev, I.info, I.lev[0].fluid), ++I.nlaunch;
    launchk(k_load_alpha<T>, nblk(g.ncell), BS, 0, I.stream, g.ncell, I.info, alpha0_dev, (T *)I.alpha), ++I.nlaunch;
    for (int l = 1; l < I.nlev; ++l) {
        Level &F = I.lev[l - 1], &Lv = I.lev[l];
        L3 LC = launch3(Lv.g);
        launchk(k_mg_fluid_coarsen, LC.grid, LC.block, 0, I.stream, to_dev(F.g), to_dev(Lv.g), F.r[0], F.r[1], F.r[2],
                                                               F.fluid, Lv.fluid), ++I.nlaunch;
    }
    OSCAR_LAUNCH_CHECK();
    // the attributes belong to the kernels, not to this instance: they are set
    // to the budget (never lowered), so that instances of other sizes, created
    // while this one runs, cannot shrink them below what this one launches with
    const void *inv = nullptr;   // FP32: static shared memory only
    if constexpr (sizeof(T) == sizeof(double))
        inv = I.g.dim == 3 ? (const void *)k_mg_inverse_band<3, T> : (const void *)k_mg_inverse_band<2, T>;
    const void *vcy = I.g.dim == 3 ? (const void *)k_mg_cluster<3, T> : (const void *)k_mg_cluster<2, T>;
    const void *sol = (const void *)k_solve_cluster<T>;
    for (const void *f : {inv, vcy, sol}) {
        if (!f) continue;
        if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClSmemBytes) != cudaSuccess ||
            cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
            return OSCAR_E_CUDA;
    }
    I.cl_fit = cluster_fit(vcy, kVcycleThreads, kVcycleCtas);
    I.solve_fit = cluster_fit(sol, 512, kMaxCluster);
    OSCAR_TRY(choose_cta(I, I.cta_cells));
    int rc = Impl<T>::interface_(I, I.alpha);
    I.nexec += I.nlaunch - l0;
    return rc;
}

template <typename T> int Solver<T>::drag_step(Instance &I, double dt) { return Impl<T>::run(I, 0, dt, 1); }

template <typename T> int Solver<T>::launch_step(Instance &I, int kind, double dt, int N) {
    int rc = Impl<T>::run_launch(I, kind, dt, N);
    if (rc) I.pending = -1;
    return rc;
}

template <typename T> int Solver<T>::finish_step(Instance &I, int *kf_out, double *test_out) {
    const int kind = I.pending, N = I.pending_N;
    int rc = Impl<T>::run_finish(I);
    if (rc == OSCAR_E_CUDA || rc == OSCAR_E_TIMEOUT) return rc;
    if (kind == 1) {
        I.last_kf = I.ctl_host[C_K];
        I.last_N = N;
        I.last_E = I.scal_host[S_E];
        I.last_dU = I.scal_host[S_DU];
    } else if (kind == 2) {
        I.last_E = I.scal_host[S_E];
        I.last_N = 1;
    }
    if (kf_out) *kf_out = kind == 1 ? I.ctl_host[C_K] : 1;
    if (test_out) *test_out = kind == 1 ? I.scal_host[S_TEST] : I.scal_host[S_E];
    return rc;
}

template <typename T> int Solver<T>::relax(Instance &I, double dt, int N, int *kf_out, double *test_out) {
    int rc = Impl<T>::run(I, 1, dt, N);
    if (rc == OSCAR_E_CUDA || rc == OSCAR_E_TIMEOUT) return rc;
    I.last_kf = I.ctl_host[C_K];
    I.last_N = N;
    I.last_E = I.scal_host[S_E];
    I.last_dU = I.scal_host[S_DU];
    if (kf_out) *kf_out = I.last_kf;
    if (test_out) *test_out = I.scal_host[S_TEST];
    return rc;
}

template <typename T> int Solver<T>::standard_step(Instance &I, double dt) {
    int rc = Impl<T>::run(I, 2, dt, 1);
    if (rc == OSCAR_E_CUDA || rc == OSCAR_E_TIMEOUT) return rc;
    I.last_E = I.scal_host[S_E];
    I.last_N = 1;
    return rc;
}

template <typename T>
__global__ void k_report_u(int n, const T *__restrict__ uvd, const double *__restrict__ usum, double invN,
                           double *__restrict__ out) {
    griddep_wait();
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < n) out[c] = (double)uvd[c] + usum[c] * invN;
}
static __global__ void k_add_pd(int n, const double *__restrict__ a, const double *__restrict__ b,
                                double *__restrict__ out) {
    griddep_wait();
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < n) out[c] = a[c] + b[c];
}

template <typename T> int Solver<T>::field_to_device(Instance &I, int which, double *dst, size_t n) {
    BlockXScope bxs(I.block_x);
    int nc = I.g.ncell;
    cudaStream_t s = I.stream;
    auto cvt = [&](const void *src, size_t len) {
        launchk(k_convert<T, double>, nblk(len), BS, 0, s, (int)len, (const T *)src, dst), ++I.nlaunch, ++I.nexec;
    };
    if (which == OSCAR_FIELD_ALPHA) cvt(I.alpha, nc);
    else if (which == OSCAR_FIELD_P) launchk(k_add_pd, nblk(nc), BS, 0, s, nc, I.p_vd, I.p_cr, dst), ++I.nlaunch, ++I.nexec;
    else if (which >= 2 && which <= 4) {
        int a = which - 2;
        if (a >= I.g.dim) cudaMemsetAsync(dst, 0, n * sizeof(double), s);
        else launchk(k_report_u<T>, nblk(nc), BS, 0, s, nc, (const T *)I.u_vd[a], I.u_sum[a], 1.0 / (double)I.last_N, dst),
                 ++I.nlaunch, ++I.nexec;
    } else if (which >= 5 && which <= 10) {
        int a = (which - 5) % 3;
        void *const *src = which < 8 ? I.u_vd : I.u_cr;
        if (a >= I.g.dim) cudaMemsetAsync(dst, 0, n * sizeof(double), s);
        else cvt(src[a], nc);
    } else if (which == OSCAR_FIELD_P_VD) cudaMemcpyAsync(dst, I.p_vd, nc * sizeof(double), cudaMemcpyDeviceToDevice, s);
    else if (which == OSCAR_FIELD_P_CR) cudaMemcpyAsync(dst, I.p_cr, nc * sizeof(double), cudaMemcpyDeviceToDevice, s);
    else if (which == OSCAR_FIELD_KAPPA) cvt(I.kappa, nc);
    else if (which >= 14 && which <= 22) {
        int a = (which - 14) % 3;
        void *const *src = which < 17 ? I.phi_vd : (which < 20 ? I.phi_cr : I.nf);
        if (a >= I.g.dim) cudaMemsetAsync(dst, 0, n * sizeof(double), s);
        else cvt(src[a], I.g.nf[a]);
    } else return OSCAR_E_INVALID_ARG;
    OSCAR_LAUNCH_CHECK();
    return 0;
}

template <typename T> int Solver<T>::field_from_device(Instance &I, int which, const double *src, size_t n) {
    BlockXScope bxs(I.block_x);
    int nc = I.g.ncell;
    cudaStream_t s = I.stream;
    auto cvt = [&](void *dst, size_t len) {
        launchk(k_convert<double, T>, nblk(len), BS, 0, s, (int)len, src, (T *)dst), ++I.nlaunch, ++I.nexec;
    };
    if (which == OSCAR_FIELD_ALPHA) {
        launchk(k_load_alpha<T>, nblk(nc), BS, 0, s, nc, I.info, src, (T *)I.alpha), ++I.nlaunch, ++I.nexec;
        OSCAR_LAUNCH_CHECK();
        long long l0 = I.nlaunch;
        int rc = Impl<T>::interface_(I, I.alpha);
        I.nexec += I.nlaunch - l0;
        return rc;
    } else if (which >= 5 && which <= 10) {
        int a = (which - 5) % 3;
        if (a >= I.g.dim) return OSCAR_E_INVALID_ARG;
        cvt(which < 8 ? I.u_vd[a] : I.u_cr[a], nc);
    } else if (which == OSCAR_FIELD_P_VD || which == OSCAR_FIELD_P) {
        cudaMemcpyAsync(I.p_vd, src, nc * sizeof(double), cudaMemcpyDeviceToDevice, s);
    } else if (which == OSCAR_FIELD_P_CR) {
        cudaMemcpyAsync(I.p_cr, src, nc * sizeof(double), cudaMemcpyDeviceToDevice, s);
    } else if (which >= 14 && which <= 19) {
        int a = (which - 14) % 3;
        if (a >= I.g.dim) return OSCAR_E_INVALID_ARG;
        cvt(which < 17 ? I.phi_vd[a] : I.phi_cr[a], I.g.nf[a]);
    } else return OSCAR_E_INVALID_ARG;
    OSCAR_LAUNCH_CHECK();
    return 0;
}

template <typename T> int Solver<T>::phase_volume(Instance &I, double *out) {
    BlockXScope bxs(I.block_x);
    launchk(k_sum_to<T>, kRedBlocks, BS, 0, I.stream, I.g.ncell, (const T *)I.alpha, I.g.V, I.partials, I.ticket, I.scal,
                                                 S_VOL), ++I.nlaunch, ++I.nexec;
    OSCAR_LAUNCH_CHECK();
    if (cudaMemcpyAsync(I.scal_host, I.scal, S_COUNT * sizeof(double), cudaMemcpyDeviceToHost, I.stream) != cudaSuccess)
        return OSCAR_E_CUDA;
    int rc = sync_bounded(I.stream, kSyncTimeoutSec);
    if (rc) return rc;
    *out = I.scal_host[S_VOL];
    return 0;
}

}  // namespace oscar
