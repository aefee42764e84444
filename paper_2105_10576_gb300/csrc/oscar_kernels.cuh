// OSCAR hot-path kernels for sm_103a (Maes & Menke, arXiv 2105.10576,
// Sections 2-3): alpha transport, interface normal and curvature, PISO
// momentum / pressure / correction, the pressure operator, CG vector
// operations and the geometric multigrid preconditioner.
//
// Every kernel is memory- or latency-bound (there is no dense contraction,
// so no tensor-core path). Layout: structure-of-arrays cell fields with x
// fastest and one face array per direction. Cell and face kernels run on 3D
// grids (x over threadIdx.x for coalesced rows, y over threadIdx.y /
// blockIdx.y, z over blockIdx.z), so no thread divides to find its cell.
// Reductions write one partial per block. The last block to finish sums them,
// or, for the dot products of the CG, every block of the kernel that needs the
// total; always in a fixed order, so every sum is deterministic run to run.
//
// Element types: T is the field type (double for the FP64 path, float for
// the mixed path); V the CG vector type (= T); the multigrid runs in T.
// FP64 arithmetic is rare on GB300 silicon, so the mixed path keeps it to the
// totals of dot products and norms (FP32 pairs below them) and the outer defect
// correction.
//
// Included by exactly one translation unit per element type.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdio.h>

#include <algorithm>
#include <utility>

#include "oscar_internal.h"

namespace oscar {

enum : int { FT_NONE = 0, FT_INTERIOR = 1, FT_WALL = 2, FT_INLET = 3, FT_OUTLET = 4 };
constexpr uint32_t INFO_FLUID = 1u << 31;
constexpr int BS = 256;
constexpr int kCtaCells = 1024;      // largest cta_cells of a schedule
constexpr int kApplyRows = 2;    // rows per thread of k_cg_pz_apply
constexpr int kUpdateRows = 4;   // rows per thread of k_cg_update
template <typename M> constexpr int kDotRows = sizeof(M) == sizeof(float) ? 2 : 1;   // rows per thread of k_mg_rbgs_dot

// Programmatic dependent launch: wait until the preceding kernel has
// completed and its writes are visible, then let the next kernel's CTAs be
// scheduled (they in turn wait here), so its launch overlaps this one.
__device__ __forceinline__ void griddep_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

__device__ __forceinline__ int ftype(uint32_t info, int a, int s) { return (info >> (3 * (2 * a + s))) & 7; }

struct GridD {
    int nx, ny, nz, ncell;
    double h[3], S[3], V;
    float hf[3], Sf[3], Vf;
};

inline GridD to_dev(const GridH &g) {
    GridD d;
    d.nx = g.nx; d.ny = g.ny; d.nz = g.nz; d.ncell = g.ncell;
    for (int a = 0; a < 3; ++a) {
        d.h[a] = g.h[a]; d.S[a] = g.S[a];
        d.hf[a] = (float)g.h[a]; d.Sf[a] = (float)g.S[a];
    }
    d.V = g.V;
    d.Vf = (float)g.V;
    return d;
}

// grid constants in the field type (no FP64 conversions in FP32 kernels)
template <typename T> struct GA;
template <> struct GA<double> {
    __device__ static __forceinline__ double h(const GridD &g, int a) { return g.h[a]; }
    __device__ static __forceinline__ double S(const GridD &g, int a) { return g.S[a]; }
};
template <> struct GA<float> {
    __device__ static __forceinline__ float h(const GridD &g, int a) { return g.hf[a]; }
    __device__ static __forceinline__ float S(const GridD &g, int a) { return g.Sf[a]; }
};

// Divisions by grid constants and the time step. An FP64 division is about ten
// FP64 instructions on a GPU that issues two FP64 FMAs per clock and SM: in
// FP64 they are multiplications by the reciprocal (GR<double>: 128x32x32 FP64
// momentum prediction 200 -> 110 us); in FP32, where they are not what bounds a
// kernel, divisions, and GR is empty.
template <typename T> struct GR {};
template <> struct GR<double> {
    double rh[3], Sh[3], rV, rS, rdt;   // 1 / h, S / h, 1 / V, 1 / (2 sum S), 1 / dt
};
template <typename T> inline GR<T> to_gr(const GridH &g, double dt) {
    GR<T> r;
    if constexpr (sizeof(T) == sizeof(double)) {
        for (int a = 0; a < 3; ++a) {
            r.rh[a] = 1.0 / g.h[a];
            r.Sh[a] = g.S[a] / g.h[a];
        }
        r.rV = 1.0 / g.V;
        r.rS = 1.0 / (2.0 * (g.S[0] + g.S[1] + g.S[2]));
        r.rdt = 1.0 / dt;
    }
    return r;
}
__device__ __forceinline__ float div_h(const GridD &g, const GR<float> &, int a, float x) { return x / g.hf[a]; }
__device__ __forceinline__ double div_h(const GridD &, const GR<double> &r, int a, double x) { return x * r.rh[a]; }
__device__ __forceinline__ double div_half_h(const GridD &, const GR<double> &r, int a, double x) { return x * (2.0 * r.rh[a]); }
__device__ __forceinline__ float mul_S_div_h(const GridD &g, const GR<float> &, int a, float x) { return x * g.Sf[a] / g.hf[a]; }
__device__ __forceinline__ double mul_S_div_h(const GridD &, const GR<double> &r, int a, double x) { return x * r.Sh[a]; }
__device__ __forceinline__ float mul_S_div_half_h(const GridD &g, const GR<float> &, int a, float x) {
    return x * g.Sf[a] / (0.5f * g.hf[a]);
}
__device__ __forceinline__ double mul_S_div_half_h(const GridD &, const GR<double> &r, int a, double x) {
    return x * (2.0 * r.Sh[a]);
}
__device__ __forceinline__ float div_V(const GridD &g, const GR<float> &, float x) { return x / g.Vf; }
__device__ __forceinline__ double div_V(const GridD &, const GR<double> &r, double x) { return x * r.rV; }
__device__ __forceinline__ float div_dt(const GR<float> &, float x, float dt) { return x / dt; }
__device__ __forceinline__ double div_dt(const GR<double> &r, double x, double) { return x * r.rdt; }
__device__ __forceinline__ float div_2S(const GR<float> &, float x, float den) { return x / den; }
__device__ __forceinline__ double div_2S(const GR<double> &r, double x, double) { return x * r.rS; }
__device__ __forceinline__ float div_by(float x, float d, float) { return x / d; }
__device__ __forceinline__ double div_by(double x, double, double rd) { return x * rd; }

template <typename T> struct P3 { T *a[3]; };
template <typename T> struct C3 { const T *a[3]; };

template <typename T> __device__ __forceinline__ T tabs(T x) { return x < T(0) ? -x : x; }

// 3D launch shape: rows of up to 256 cells along x, several rows per block
// when rows are short.
struct L3 {
    dim3 grid, block;
    int nblocks;
};
inline L3 launch3(int nx, int ny, int nz) {
    int bx = nx >= 256 ? 256 : (nx > 64 ? 128 : (nx > 32 ? 64 : 32));
    if (t_block_x > 0 && t_block_x < bx) bx = t_block_x;   // the instance's schedule caps the x extent
    int by = BS / bx;
    L3 l;
    l.block = dim3(bx, by, 1);
    l.grid = dim3((nx + bx - 1) / bx, (ny + by - 1) / by, nz);
    l.nblocks = (int)(l.grid.x * l.grid.y * l.grid.z);
    return l;
}
inline L3 launch3(const GridH &g) { return launch3(g.nx, g.ny, g.nz); }
inline L3 launch3_faces(const GridH &g, int a) { return launch3(g.nx + (a == 0), g.ny + (a == 1), g.nz + (a == 2)); }
// blocks of launch3's shape over (x, rows); about target blocks, each thread
// taking m rows (ROW_LOOP)
inline L3 launch_rows(const GridH &g, int target) {
    L3 l = launch3(g.nx, g.ny * g.nz, 1);
    int gx = (int)l.grid.x, gy = (int)l.grid.y;
    int want = target / gx > 0 ? target / gx : 1;
    int m = (gy + want - 1) / want;
    l.grid = dim3(gx, (gy + m - 1) / m, 1);
    l.nblocks = (int)(l.grid.x * l.grid.y);
    return l;
}

// at most two blocks of 1024 threads per SM over (x, rows), rows looped
inline L3 launch_sms(const GridH &g) {
    L3 l = launch3(g.nx, g.ny * g.nz, 1);
    const int bx = (int)l.block.x, by = 1024 / bx, gx = (int)l.grid.x, gy = (g.ny * g.nz + by - 1) / by;
    l.block = dim3(bx, by, 1);
    l.grid = dim3(gx, std::max(1, std::min(gy, 304 / gx)), 1);
    l.nblocks = (int)(l.grid.x * l.grid.y);
    return l;
}

#define CELL_IJK(g)                                            \
    const int i = blockIdx.x * blockDim.x + threadIdx.x;       \
    const int j = blockIdx.y * blockDim.y + threadIdx.y;       \
    const int k = blockIdx.z;                                  \
    const bool inside = i < (g).nx && j < (g).ny;              \
    const int c = i + (g).nx * (j + (g).ny * k);

#define BLOCK_ID() ((int)(blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z)))

// Blocks of launch3's shape over (x, rows) where each thread takes rpt rows of a
// group, row = group * blockDim.y * rpt + threadIdx.y + u * blockDim.y, u < rpt
// (the kernels unroll u so that the loads of all their rows are in flight
// together). At most kDotBlocks blocks and one more per column of blocks: a
// block takes the groups blockIdx.y, blockIdx.y + gridDim.y, ...
constexpr int kDotBlocks = 608;   // 152 SMs x 4
struct L3G : L3 { int groups; };
inline L3G launch_groups(int nx, int rows, int rpt) {
    L3G l;
    static_cast<L3 &>(l) = launch3(nx, rows, 1);
    const int by = (int)l.block.y, gx = (int)l.grid.x;
    l.groups = (rows + by * rpt - 1) / (by * rpt);
    const int m = std::max(1, (int)(((long long)l.groups * gx + kDotBlocks - 1) / kDotBlocks));
    l.grid = dim3(gx, (l.groups + m - 1) / m, 1);
    l.nblocks = (int)(l.grid.x * l.grid.y);
    return l;
}

// Row loop of the stencil reductions (launch_rows): the thread at x = i takes
// every (gridDim.y * blockDim.y)-th row, row = j + ny k, so that a thread sums
// several cells before the block reduction.
#define ROW_LOOP(g)                                              \
    const int i = blockIdx.x * blockDim.x + threadIdx.x;         \
    const int nrow_ = (g).ny * (g).nz;                           \
    for (int row = blockIdx.y * blockDim.y + threadIdx.y; row < nrow_; row += gridDim.y * blockDim.y)
#define ROW_CELL(g)                                              \
    const int k = row / (g).ny, j = row - k * (g).ny;            \
    const int c = i + (g).nx * row;

__device__ __forceinline__ int flo(const GridD &g, int a, int i, int j, int k) {
    if (a == 0) return i + (g.nx + 1) * (j + g.ny * k);
    if (a == 1) return i + g.nx * (j + (g.ny + 1) * k);
    return i + g.nx * (j + g.ny * k);
}
__device__ __forceinline__ int fhi(const GridD &g, int a, int i, int j, int k) {
    if (a == 0) return flo(g, 0, i, j, k) + 1;
    if (a == 1) return flo(g, 1, i, j, k) + g.nx;
    return flo(g, 2, i, j, k) + g.nx * g.ny;
}
__device__ __forceinline__ int noff(const GridD &g, int a) { return a == 0 ? 1 : (a == 1 ? g.nx : g.nx * g.ny); }

// Face kernels: thread (i,j,k) of the face grid of direction A; the face
// sits on the low side of cell (i,j,k).
#define FACE_IJK(g, A)                                                   \
    const int i = blockIdx.x * blockDim.x + threadIdx.x;                 \
    const int j = blockIdx.y * blockDim.y + threadIdx.y;                 \
    const int k = blockIdx.z;                                            \
    const int fnx = (g).nx + ((A) == 0), fny = (g).ny + ((A) == 1);      \
    if (i >= fnx || j >= fny) return;                                    \
    const int f = i + fnx * (j + fny * k);

// Fluid neighbours and type of the face of direction A at face coordinates
// (i,j,k).
template <int A>
__device__ __forceinline__ int decode_face(const GridD &g, const uint32_t *__restrict__ info, int i, int j, int k,
                                           int &L, int &H) {
    const int q = A == 0 ? i : (A == 1 ? j : k);
    const int n = A == 0 ? g.nx : (A == 1 ? g.ny : g.nz);
    const int off = A == 0 ? 1 : (A == 1 ? g.nx : g.nx * g.ny);
    const int c = i + g.nx * (j + g.ny * k);
    L = -1; H = -1;
    if (q < n && (info[c] & INFO_FLUID)) {
        int t = ftype(info[c], A, 0);
        H = c;
        if (t == FT_INTERIOR) L = c - off;
        return t;
    }
    if (q > 0 && (info[c - off] & INFO_FLUID)) {
        L = c - off;
        return ftype(info[c - off], A, 1);
    }
    return FT_NONE;
}

// ---------------------------------------------------------------------------
// reductions (one partial per block, finished in one block: deterministic)
// ---------------------------------------------------------------------------
// Block reductions, deterministic, result valid in thread 0. The per-thread
// values pass through shared memory and only warp 0 does FP64 arithmetic:
// GB300 issues FP64 at a small fraction of its FP32 rate, and a shuffle tree
// in every warp made FP64 the bottleneck of the vector kernels.
__device__ __forceinline__ double block_reduce(double v, bool is_max) {
    __shared__ double sh[1024];
    const int t = threadIdx.x + blockDim.x * threadIdx.y, nt = blockDim.x * blockDim.y;
    __syncthreads();   // a previous reduction's readers are done with sh
    sh[t] = v;
    __syncthreads();
    if (t < 32) {
        double s = t < nt ? sh[t] : 0.0;
        for (int q = t + 32; q < nt; q += 32) s = is_max ? fmax(s, sh[q]) : s + sh[q];
        for (int o = 16; o > 0; o >>= 1) {
            double w = __shfl_down_sync(0xffffffffu, s, o);
            s = is_max ? fmax(s, w) : s + w;
        }
        v = s;
    }
    return v;
}
__device__ __forceinline__ double block_sum(double v) { return block_reduce(v, false); }
__device__ __forceinline__ double block_max(double v) { return block_reduce(v, true); }
// Compensated block sums of FP32 values: the (sum, rounding error) pair is
// carried through the shuffle tree with error-free TwoSum steps (Knuth), so
// the block total matches the FP64 sum of the thread values to about 2^-44
// relative, with FP32 instructions only.
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}
__device__ __forceinline__ void warp_sum_pair(float &s, float &e) {
    for (int o = 16; o > 0; o >>= 1) {
        const float so = __shfl_down_sync(0xffffffffu, s, o), eo = __shfl_down_sync(0xffffffffu, e, o);
        float t, err;
        two_sum(s, so, t, err);
        s = t;
        e += eo + err;
    }
}
// block total of compensated pairs (s, e); the result is valid in thread 0
__device__ __forceinline__ void block_pair_f(float &s, float &e) {
    __shared__ float shs[32], she[32];
    const int t = threadIdx.x + blockDim.x * threadIdx.y, nt = blockDim.x * blockDim.y;
    const int w = t >> 5, l = t & 31, nw = nt >> 5;
    warp_sum_pair(s, e);
    __syncthreads();
    if (l == 0) { shs[w] = s; she[w] = e; }
    __syncthreads();
    if (w == 0) {
        s = l < nw ? shs[l] : 0.f;
        e = l < nw ? she[l] : 0.f;
        warp_sum_pair(s, e);
    }
}
__device__ __forceinline__ bool block_leader() { return threadIdx.x == 0 && threadIdx.y == 0; }

// Single-pass reduction: every block stores its partial(s); the block that
// finishes last (atomic ticket) sums all partials in block order and returns
// true with the totals in v0 / v1 (all its threads). Deterministic, no spin.
// Every thread of every block must call it.
__device__ __forceinline__ bool reduce_last(double &v0, double &v1, int nv, bool is_max, double *__restrict__ part,
                                            int stride, unsigned *__restrict__ ticket, int nb) {
    v0 = is_max ? block_max(v0) : block_sum(v0);
    if (nv > 1) v1 = block_sum(v1);
    __shared__ int last_s;
    __shared__ double tot_s[2];
    if (block_leader()) {
        int b = BLOCK_ID();
        part[b] = v0;
        if (nv > 1) part[stride + b] = v1;
        __threadfence();
        unsigned t = atomicAdd(ticket, 1u);
        last_s = (t == (unsigned)(nb - 1)) ? 1 : 0;
    }
    __syncthreads();
    if (!last_s) return false;
    __threadfence();
    int tid = threadIdx.x + blockDim.x * threadIdx.y, nt = blockDim.x * blockDim.y;
    double s0 = 0.0, s1 = 0.0;
    for (int b = tid; b < nb; b += nt) {
        double p0 = __ldcg(part + b);
        s0 = is_max ? fmax(s0, p0) : s0 + p0;
        if (nv > 1) s1 += __ldcg(part + stride + b);
    }
    s0 = is_max ? block_max(s0) : block_sum(s0);
    if (nv > 1) s1 = block_sum(s1);
    if (block_leader()) {
        tot_s[0] = s0;
        tot_s[1] = s1;
        *ticket = 0u;
    }
    __syncthreads();
    v0 = tot_s[0];
    v1 = tot_s[1];
    return true;
}

// reduce_last for up to four FP64 sums (v[0 .. nv), partial slots q * stride),
// each summed as reduce_last sums one
__device__ __forceinline__ bool reduce_last4(double *v, int nv, double *__restrict__ part, int stride,
                                             unsigned *__restrict__ ticket, int nb) {
    for (int q = 0; q < nv; ++q) v[q] = block_sum(v[q]);
    __shared__ int last_s;
    __shared__ double tot_s[4];
    if (block_leader()) {
        int b = BLOCK_ID();
        for (int q = 0; q < nv; ++q) part[q * stride + b] = v[q];
        __threadfence();
        unsigned t = atomicAdd(ticket, 1u);
        last_s = (t == (unsigned)(nb - 1)) ? 1 : 0;
    }
    __syncthreads();
    if (!last_s) return false;
    __threadfence();
    int tid = threadIdx.x + blockDim.x * threadIdx.y, nt = blockDim.x * blockDim.y;
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    for (int b = tid; b < nb; b += nt)
        for (int q = 0; q < nv; ++q) s[q] += __ldcg(part + q * stride + b);
    for (int q = 0; q < nv; ++q) s[q] = block_sum(s[q]);
    if (block_leader()) {
        for (int q = 0; q < nv; ++q) tot_s[q] = s[q];
        *ticket = 0u;
    }
    __syncthreads();
    for (int q = 0; q < nv; ++q) v[q] = tot_s[q];
    return true;
}

// Dot products of the CG. A thread sums groups of cells in the vectors' type
// (the groups of its kernel) and the groups in compensated pairs (FP32) or
// plainly (FP64); a block stores one partial and ends. The kernel that needs
// the total sums the partials itself, every block in the same order, beside
// its own loads. That leaves out a finishing block: a fence and an atomic in
// every block, 1.4 us, and a last block that sums 2048 partials alone while
// the next kernel waits, 2.8 us of the 9.2 us of the r.z sweep at 256x64x64.
// With at most about kDotBlocks partials a thread of a 256-thread block loads
// three.
struct DotAcc64 {
    double s = 0.0;
    __device__ __forceinline__ void add(double v) { s += v; }
};
struct DotAcc32 {
    float s = 0.f, e = 0.f;
    __device__ __forceinline__ void add(float v) {
        float sn, se;
        two_sum(s, v, sn, se);
        s = sn;
        e += se;
    }
};
template <typename V> struct DotAcc { using type = DotAcc64; };
template <> struct DotAcc<float> { using type = DotAcc32; };
__device__ __forceinline__ void dot_store(DotAcc32 a, double *part) {
    block_pair_f(a.s, a.e);
    if (block_leader()) reinterpret_cast<float2 *>(part)[BLOCK_ID()] = make_float2(a.s, a.e);
}
__device__ __forceinline__ void dot_store(DotAcc64 a, double *part) {
    const double v = block_sum(a.s);
    if (block_leader()) part[BLOCK_ID()] = v;
}
// total of nb partials of vectors of type V, valid in the block leader (every
// thread calls it)
template <typename V> __device__ __forceinline__ double dot_total(const double *part, int nb);
template <> __device__ __forceinline__ double dot_total<float>(const double *part, int nb) {
    const int nt = blockDim.x * blockDim.y, t = threadIdx.x + blockDim.x * threadIdx.y;
    float s = 0.f, e = 0.f;
    for (int q = t; q < nb; q += nt) {
        const float2 v = __ldcg(reinterpret_cast<const float2 *>(part) + q);
        float sn, se;
        two_sum(s, v.x, sn, se);
        s = sn;
        e += se + v.y;
    }
    block_pair_f(s, e);
    return (double)s + (double)e;
}
template <> __device__ __forceinline__ double dot_total<double>(const double *part, int nb) {
    const int nt = blockDim.x * blockDim.y, t = threadIdx.x + blockDim.x * threadIdx.y;
    double s = 0.0;
    for (int q = t; q < nb; q += nt) s += __ldcg(part + q);
    return block_sum(s);
}

// Loop-control decisions taken by the finishing block: each writes
// ctl[C_COND] and, inside a graph, the conditional handle.
__device__ __forceinline__ void set_cond(int *ctl, cudaGraphConditionalHandle h, bool more) {
    ctl[C_COND] = more ? 1 : 0;
    if (h) cudaGraphSetConditional(h, more ? 1u : 0u);
}

// after r = b - M q: mode 0 = start of a plain PCG solve; 1 / 2 = first /
// later check of the defect-correction loop (mixed path)
constexpr int kMaxOuter = 40;          // defect-correction trips (mixed path)
constexpr double kInnerRtol = 1e-4;    // FP32 inner solve: residual reduction per trip
constexpr double kTripMargin = 0.5;    // ... or down to this fraction of the outer target
__device__ __forceinline__ void residual_control(double *scal, int *ctl, double rtol, int mode,
                                                 cudaGraphConditionalHandle h) {
    double bn = sqrt(scal[S_BB]), rn = sqrt(scal[S_RR]);
    bool bad = !(isfinite(bn) && isfinite(rn));
    if (bad) ctl[C_NAN] = 1;
    if (mode == 0) {
        double target = rtol * (bn > 0.0 ? bn : rn);
        scal[S_TARGET] = target;
        scal[S_RZ0] = 0.0;
        ctl[C_IT] = 0;
        set_cond(ctl, h, !bad && rn > target);
        return;
    }
    scal[S_RZ0] = 0.0;   // the FP32 iteration starts afresh
    ctl[C_IT] = 0;
    if (mode == 1) {
        scal[S_TARGET] = rtol * (bn > 0.0 ? bn : rn);
        ctl[C_OUT] = 0;
    } else {
        ctl[C_OUT] += 1;
        ctl[C_OSUM] += 1;
    }
    bool more = !bad && rn > scal[S_TARGET];
    if (more && ctl[C_OUT] >= kMaxOuter) { ctl[C_NOTCONV] = 1; more = false; }
    // the FP32 trip stops at kInnerRtol times its starting residual, or as
    // soon as half the outer target is reached (solving below what the FP64
    // test asks for is wasted; the factor 2 covers the drift of the FP32
    // recursive residual from the true one, and a trip that still ends above
    // the target is followed by another)
    scal[S_ITARGET] = fmax(kInnerRtol * rn, kTripMargin * scal[S_TARGET]);
    set_cond(ctl, h, more);
}


// ---------------------------------------------------------------------------
// set-up
// ---------------------------------------------------------------------------
template <int DIM>
__global__ void k_build_info(GridD g, const uint8_t *__restrict__ solid, uint32_t *__restrict__ info,
                             uint8_t *__restrict__ fluid) {
    griddep_wait();
    CELL_IJK(g);
    if (!inside) return;
    if (solid[c]) { info[c] = 0; fluid[c] = 0; return; }
    int ijk[3] = {i, j, k};
    int n[3] = {g.nx, g.ny, g.nz};
    uint32_t w = INFO_FLUID;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        for (int s = 0; s < 2; ++s) {
            int q = ijk[a] + (s ? 1 : -1);
            int t;
            if (q < 0) t = (a == 0) ? FT_INLET : FT_WALL;
            else if (q >= n[a]) t = (a == 0) ? FT_OUTLET : FT_WALL;
            else t = solid[c + (s ? 1 : -1) * noff(g, a)] ? FT_WALL : FT_INTERIOR;
            w |= (uint32_t)t << (3 * (2 * a + s));
        }
    }
    info[c] = w;
    fluid[c] = 1;
}

template <typename T>
__global__ void k_load_alpha(int n, const uint32_t *__restrict__ info, const double *__restrict__ src, T *__restrict__ dst) {
    griddep_wait();
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n) return;
    dst[c] = (info[c] & INFO_FLUID) ? (T)src[c] : T(0);
}

template <typename S, typename D>
__global__ void k_convert(int n, const S *__restrict__ src, D *__restrict__ dst) {
    griddep_wait();
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < n) dst[c] = (D)src[c];
}

template <typename T>
__global__ void k_sum2(int n, const T *__restrict__ a, const T *__restrict__ b, T *__restrict__ out) {
    griddep_wait();
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < n) out[c] = a[c] + b[c];
}

// ---------------------------------------------------------------------------
// alpha transport: explicit Euler (Eq. alphaExp) with a vanLeer high-order
// flux, interface compression and a Zalesak flux-corrected-transport limiter
// ---------------------------------------------------------------------------
// Low-order (upwind) flux FL and antidiffusive flux AD of an interior face
// between fluid cells L (low) and H (high) of direction a.
template <typename T>
__device__ __forceinline__ void ho_flux(const uint32_t *__restrict__ info, const T *__restrict__ alpha, int a, int off,
                                        int L, int H, T ph, T nfv, T c_alpha, T &FL, T &AD) {
    int U, D, UU = -1;
    if (ph >= T(0)) {
        U = L; D = H;
        if (ftype(info[L], a, 0) == FT_INTERIOR) UU = L - off;
    } else {
        U = H; D = L;
        if (ftype(info[H], a, 1) == FT_INTERIOR) UU = H + off;
    }
    T aU = alpha[U], aD = alpha[D];
    T dc = aD - aU;
    T du = UU >= 0 ? (aU - alpha[UU]) : T(0);
    // vanLeer: aU + psi(r)/2 (aD - aU), psi = (r+|r|)/(1+|r|), r = du/dc
    T avl = (du * dc > T(0)) ? aU + du * dc / (du + dc) : aU;
    T flow = ph * aU;
    // compression flux phi_r alpha (1 - alpha), phi_r = c_alpha |phi| n_f
    T phir = c_alpha * tabs(ph) * nfv;
    T aLv = alpha[L], aHv = alpha[H];
    T fc = (phir >= T(0)) ? phir * aLv * (T(1) - aHv) : phir * aHv * (T(1) - aLv);
    T fhigh = ph * avl + fc;
    FL = flow;
    AD = fhigh - flow;
}

template <int DIM, typename T>
__global__ void k_transport_low(GridD g, const uint32_t *__restrict__ info, const T *__restrict__ alpha, C3<T> phi,
                                C3<T> nf, T c_alpha, T alpha_in, T rV, T *__restrict__ aL, T *__restrict__ Pp,
                                T *__restrict__ Pm) {
    griddep_wait();
    CELL_IJK(g);
    if (!inside) return;
    uint32_t inf = info[c];
    if (!(inf & INFO_FLUID)) { aL[c] = T(0); Pp[c] = T(0); Pm[c] = T(0); return; }
    T out = T(0), pp = T(0), pm = T(0);
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        int off = noff(g, a);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            int t = ftype(inf, a, s);
            int f = s ? fhi(g, a, i, j, k) : flo(g, a, i, j, k);
            T ph = phi.a[a][f];
            T FL = T(0), AD = T(0);
            if (t == FT_INTERIOR) {
                int nb = s ? c + off : c - off;
                ho_flux<T>(info, alpha, a, off, s ? c : nb, s ? nb : c, ph, nf.a[a][f], c_alpha, FL, AD);
            } else if (t == FT_INLET) {
                FL = ph >= T(0) ? ph * alpha_in : ph * alpha[c];
            } else if (t == FT_OUTLET) {
                FL = ph * alpha[c];
            }
            out += s ? FL : -FL;
            T aout = s ? AD : -AD;
            if (aout > T(0)) pm += aout; else pp += -aout;
        }
    }
    aL[c] = alpha[c] - rV * out;
    Pp[c] = pp;
    Pm[c] = pm;
}

template <int DIM, typename T>
__global__ void k_transport_ratio(GridD g, const uint32_t *__restrict__ info, const T *__restrict__ alpha,
                                  const T *__restrict__ aL, const T *__restrict__ Pp, const T *__restrict__ Pm, T rV,
                                  T rrV, T *__restrict__ Rp, T *__restrict__ Rm) {
    griddep_wait();
    CELL_IJK(g);
    if (!inside) return;
    uint32_t inf = info[c];
    if (!(inf & INFO_FLUID)) { Rp[c] = T(0); Rm[c] = T(0); return; }
    T a0 = alpha[c], l0 = aL[c];
    T amax = a0 > l0 ? a0 : l0;
    T amin = a0 < l0 ? a0 : l0;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        int off = noff(g, a);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            if (ftype(inf, a, s) != FT_INTERIOR) continue;
            int nb = s ? c + off : c - off;
            T an = alpha[nb], ln = aL[nb];
            if (an > amax) amax = an;
            if (ln > amax) amax = ln;
            if (an < amin) amin = an;
            if (ln < amin) amin = ln;
        }
    }
    if (amax > T(1)) amax = T(1);
    if (amin < T(0)) amin = T(0);
    T Qp = div_by(amax - l0, rV, rrV);
    T Qm = div_by(l0 - amin, rV, rrV);
    if (Qp < T(0)) Qp = T(0);
    if (Qm < T(0)) Qm = T(0);
    T pp = Pp[c], pm = Pm[c];
    Rp[c] = pp > T(0) ? (Qp / pp < T(1) ? Qp / pp : T(1)) : T(0);
    Rm[c] = pm > T(0) ? (Qm / pm < T(1) ? Qm / pm : T(1)) : T(0);
}

template <int DIM, typename T>
__global__ void k_transport_update(GridD g, const uint32_t *__restrict__ info, const T *__restrict__ alpha, C3<T> phi,
                                   C3<T> nf, T c_alpha, const T *__restrict__ aL, const T *__restrict__ Rp,
                                   const T *__restrict__ Rm, T rV, T *__restrict__ alpha_new) {
    griddep_wait();
    CELL_IJK(g);
    if (!inside) return;
    uint32_t inf = info[c];
    if (!(inf & INFO_FLUID)) { alpha_new[c] = T(0); return; }
    T out = T(0);
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        int off = noff(g, a);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            if (ftype(inf, a, s) != FT_INTERIOR) continue;
            int f = s ? fhi(g, a, i, j, k) : flo(g, a, i, j, k);
            int nb = s ? c + off : c - off;
            int L = s ? c : nb, H = s ? nb : c;
            T FL, AD;
            ho_flux<T>(info, alpha, a, off, L, H, phi.a[a][f], nf.a[a][f], c_alpha, FL, AD);
            T lam;
            if (AD >= T(0)) lam = Rm[L] < Rp[H] ? Rm[L] : Rp[H];
            else lam = Rm[H] < Rp[L] ? Rm[H] : Rp[L];
            T fl = lam * AD;
            out += s ? fl : -fl;
        }
    }
    alpha_new[c] = aL[c] - rV * out;
}

// ---------------------------------------------------------------------------
// interface: smoothed alpha, face normals with the contact angle, curvature
// (Section 2.1; wall condition of Eqs. VOFd / VOFc)
// ---------------------------------------------------------------------------
template <int DIM, typename T>
__global__ void k_smooth(GridD g, GR<T> gr, const uint32_t *__restrict__ info, const T *__restrict__ src, T *__restrict__ dst) {
    griddep_wait();
    CELL_IJK(g);
    if (!inside) return;
    uint32_t inf = info[c];
    if (!(inf & INFO_FLUID)) { dst[c] = T(0); return; }
    T num = T(0), den = T(0);
    T x = src[c];
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        int off = noff(g, a);
        T Sa = GA<T>::S(g, a);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            T af = ftype(inf, a, s) == FT_INTERIOR ? T(0.5) * (x + src[s ? c + off : c - off]) : x;
            num += af * Sa;
            den += Sa;
        }
    }
    dst[c] = div_2S(gr, num, den);
}

template <int DIM, typename T>
__device__ __forceinline__ T gauss_grad(const GridD &g, const GR<T> &gr, const uint32_t *__restrict__ info, const T *__restrict__ x, int c,
                                        int b) {
    uint32_t inf = info[c];
    int off = noff(g, b);
    T xc = x[c];
    T f0 = ftype(inf, b, 0) == FT_INTERIOR ? T(0.5) * (xc + x[c - off]) : xc;
    T f1 = ftype(inf, b, 1) == FT_INTERIOR ? T(0.5) * (xc + x[c + off]) : xc;
    return div_h(g, gr, b, f1 - f0);
}

template <int DIM, int A, typename T>
__global__ void k_normals(GridD g, GR<T> gr, const uint32_t *__restrict__ info, const T *__restrict__ as, T ct, T deltaN,
                          T *__restrict__ nfA) {
    griddep_wait();
    FACE_IJK(g, A);
    int L, H;
    int t = decode_face<A>(g, info, i, j, k, L, H);
    T n = T(0);
    if (t == FT_INTERIOR) {
        T gv[3] = {T(0), T(0), T(0)};
        gv[A] = div_h(g, gr, A, as[H] - as[L]);
#pragma unroll
        for (int b = 0; b < DIM; ++b) {
            if (b == A) continue;
            gv[b] = T(0.5) * (gauss_grad<DIM, T>(g, gr, info, as, L, b) + gauss_grad<DIM, T>(g, gr, info, as, H, b));
        }
        T mag = T(0);
#pragma unroll
        for (int b = 0; b < DIM; ++b) mag += gv[b] * gv[b];
        mag = sqrt(mag);
        n = gv[A] / (mag + deltaN);
    } else if (t == FT_WALL) {
        n = (L >= 0) ? ct : -ct;   // n . n_wall = cos(theta), n_wall out of the fluid cell
    }
    nfA[f] = n;
}

template <int DIM, typename T>
__global__ void k_curvature(GridD g, GR<T> gr, const uint32_t *__restrict__ info, C3<T> nf, T *__restrict__ kappa) {
    griddep_wait();
    CELL_IJK(g);
    if (!inside) return;
    if (!(info[c] & INFO_FLUID)) { kappa[c] = T(0); return; }
    T acc = T(0);
#pragma unroll
    for (int a = 0; a < DIM; ++a) acc += div_h(g, gr, a, nf.a[a][fhi(g, a, i, j, k)] - nf.a[a][flo(g, a, i, j, k)]);
    kappa[c] = -acc;
}

// ---------------------------------------------------------------------------
// PISO (Section 2.2 with Eqs. NSE1d / NSEc, advective form of ddt + convection)
// ---------------------------------------------------------------------------
template <typename T> struct Fluid { T rho1, rho2, mu1, mu2; };
template <typename T> __device__ __forceinline__ T mix(T al, T p1, T p2) { return al * p1 + (T(1) - al) * p2; }

// Mechanical energy of the relaxation: the interfacial energy sigma A, with
// A = sum over fluid cells of |grad alpha| V (Gauss gradient, boundary faces
// take the cell's value), plus the kinetic energy sum of rho(alpha) |u|^2 V / 2.
// The finishing block stores it in scal[slot]. Section 6 suggests identifying
// capillary equilibrium by an energy balance; the relaxation's
// OSCAR_CONV_AREA mode exits when this energy changes by less than the
// tolerance (relative) over a sub-step.
template <int DIM, typename T>
__global__ void k_relax_energy(int n, GridD g, GR<T> gr, const uint32_t *__restrict__ info, const T *__restrict__ alpha,
                               C3<T> u, Fluid<T> fl, double sigma, double *__restrict__ part, int stride,
                               unsigned *__restrict__ ticket, double *__restrict__ scal, int slot) {
    griddep_wait();
    double area = 0.0, kin = 0.0;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) {
        if (!(info[c] & INFO_FLUID)) continue;
        T m2 = T(0), u2 = T(0);
#pragma unroll
        for (int b = 0; b < DIM; ++b) {
            const T gb = gauss_grad<DIM, T>(g, gr, info, alpha, c, b);
            m2 += gb * gb;
            const T ub = u.a[b][c];
            u2 += ub * ub;
        }
        area += (double)sqrt(m2) * g.V;
        kin += 0.5 * (double)mix(alpha[c], fl.rho1, fl.rho2) * (double)u2 * g.V;
    }
    if (reduce_last(area, kin, 2, false, part, stride, ticket, gridDim.x) && block_leader())
        scal[slot] = sigma * area + kin;
}

// rA = 1/A, A = rho/dt + (viscous diagonal + rho * inflow flux)/V
template <int DIM, typename T>
__global__ void k_rA(GridD g, GR<T> gr, const uint32_t *__restrict__ info, const T *__restrict__ alpha, C3<T> phic, Fluid<T> fl,
                     T dt, T *__restrict__ rA) {
    griddep_wait();
    CELL_IJK(g);
    if (!inside) return;
    uint32_t inf = info[c];
    if (!(inf & INFO_FLUID)) { rA[c] = T(0); return; }
    T al = alpha[c];
    T rho = mix(al, fl.rho1, fl.rho2), mu = mix(al, fl.mu1, fl.mu2);
    T acc = T(0), cin = T(0);
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        int off = noff(g, a);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            int t = ftype(inf, a, s);
            if (t == FT_INTERIOR) {
                T mun = mix(alpha[s ? c + off : c - off], fl.mu1, fl.mu2);
                acc += mul_S_div_h(g, gr, a, T(0.5) * (mu + mun));
            } else if (t == FT_WALL || t == FT_INLET) {
                acc += mul_S_div_half_h(g, gr, a, mu);
            }
            if (t == FT_INTERIOR || t == FT_INLET) {
                T fo = (s ? T(1) : T(-1)) * phic.a[a][s ? fhi(g, a, i, j, k) : flo(g, a, i, j, k)];
                if (fo < T(0)) cin += -fo;   // inflow: implicit upwind part of convection
            }
        }
    }
    rA[c] = T(1) / (div_dt(gr, rho, dt) + div_V(g, gr, acc + rho * cin));
}

// pressure-operator coefficients c_f (multigrid level 0) and CSF face forces
template <int A, typename T>
__global__ void k_face_coeffs(GridD g, GR<T> gr, const uint32_t *__restrict__ info, const T *__restrict__ rA,
                              const T *__restrict__ kappa, const T *__restrict__ alpha, T sigma, int has_st,
                              T *__restrict__ cf, T *__restrict__ fst, double *__restrict__ cf64) {
    griddep_wait();
    FACE_IJK(g, A);
    int L, H;
    int t = decode_face<A>(g, info, i, j, k, L, H);
    T cc = T(0), fs = T(0);
    if (t == FT_INTERIOR) {
        cc = mul_S_div_h(g, gr, A, T(0.5) * (rA[L] + rA[H]));
        if (has_st) fs = div_h(g, gr, A, sigma * T(0.5) * (kappa[L] + kappa[H]) * (alpha[H] - alpha[L]));
    } else if (t == FT_OUTLET) {
        cc = mul_S_div_half_h(g, gr, A, rA[L]);
    }
    cf[f] = cc;
    fst[f] = fs;
    if (cf64) cf64[f] = (double)cc;
}

// Gauss gradients of the velocity iterate: G[comp*3 + dir]
template <int DIM, typename T>
__global__ void k_vel_grad(GridD g, GR<T> gr, const uint32_t *__restrict__ info, C3<T> v, T vin0, P3<T> G0, P3<T> G1, P3<T> G2) {
    griddep_wait();
    CELL_IJK(g);
    if (!inside) return;
    uint32_t inf = info[c];
    if (!(inf & INFO_FLUID)) return;
    T *Gr[3][3] = {{G0.a[0], G0.a[1], G0.a[2]}, {G1.a[0], G1.a[1], G1.a[2]}, {G2.a[0], G2.a[1], G2.a[2]}};
#pragma unroll
    for (int comp = 0; comp < DIM; ++comp) {
        T vc = v.a[comp][c];
        T vin = comp == 0 ? vin0 : T(0);
#pragma unroll
        for (int dir = 0; dir < DIM; ++dir) {
            int off = noff(g, dir);
            T fv[2];
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                int t = ftype(inf, dir, s);
                if (t == FT_INTERIOR) fv[s] = T(0.5) * (vc + v.a[comp][s ? c + off : c - off]);
                else if (t == FT_INLET) fv[s] = vin;
                else if (t == FT_OUTLET) fv[s] = vc;
                else fv[s] = T(0);
            }
            Gr[comp][dir][c] = div_h(g, gr, dir, fv[1] - fv[0]);
        }
    }
}

// HbyA = H/A: old-time term, neighbour part of the viscous Laplacian, inflow
// (implicit upwind) neighbours, explicit linear-upwind correction and the
// transpose viscous term. A latency-bound gather: the register cap (6 blocks
// of 256 threads per SM instead of 4) keeps more loads in flight.
template <int DIM, typename T>
__global__ void __launch_bounds__(256, 6) k_momentum_H(GridD g, GR<T> gr, const uint32_t *__restrict__ info, C3<T> v, C3<T> vold, C3<T> phic,
                             const T *__restrict__ alpha, const T *__restrict__ rA, Fluid<T> fl, T vin0, T dt,
                             C3<T> G0, C3<T> G1, C3<T> G2, P3<T> hbya) {
    griddep_wait();
    CELL_IJK(g);
    if (!inside) return;
    uint32_t inf = info[c];
    if (!(inf & INFO_FLUID)) {
#pragma unroll
        for (int comp = 0; comp < DIM; ++comp) hbya.a[comp][c] = T(0);
        return;
    }
    const T *Gr[3][3] = {{G0.a[0], G0.a[1], G0.a[2]}, {G1.a[0], G1.a[1], G1.a[2]}, {G2.a[0], G2.a[1], G2.a[2]}};
    T al = alpha[c];
    T rho = mix(al, fl.rho1, fl.rho2), mu = mix(al, fl.mu1, fl.mu2);
    T rAc = rA[c];
    T lap[3] = {T(0), T(0), T(0)}, conv[3] = {T(0), T(0), T(0)}, tr[3] = {T(0), T(0), T(0)},
      inflow[3] = {T(0), T(0), T(0)};
    T vc[3];
#pragma unroll
    for (int comp = 0; comp < DIM; ++comp) vc[comp] = v.a[comp][c];
    // faces outer, components inner: the face type, neighbour, flux, face
    // viscosity and upwind cell are worked out once per face
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        const int off = noff(g, a);
        const T Sa = GA<T>::S(g, a), ha = GA<T>::h(g, a);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int t = ftype(inf, a, s);
            const T sg = s ? T(1) : T(-1);
            const int f = s ? fhi(g, a, i, j, k) : flo(g, a, i, j, k);
            if (t == FT_INTERIOR) {
                const int nb = s ? c + off : c - off;
                const T mun = mix(alpha[nb], fl.mu1, fl.mu2);
                const T muf = T(0.5) * (mu + mun);
                const T lapc = mul_S_div_h(g, gr, a, muf);
                const T pc = phic.a[a][f];
                const bool fromL = pc >= T(0);
                const int up = fromL ? (s ? c : nb) : (s ? nb : c);
                const T hs = fromL ? T(0.5) * ha : -(T(0.5) * ha);
                const T fo = sg * pc;
                const T trc = sg * muf * Sa;
#pragma unroll
                for (int comp = 0; comp < DIM; ++comp) {
                    const T vn = v.a[comp][nb];
                    lap[comp] += lapc * vn;
                    const T vu = fromL ? (s ? vc[comp] : vn) : (s ? vn : vc[comp]);
                    const T vf = vu + hs * Gr[comp][a][up];
                    if (fo < T(0)) inflow[comp] += -fo * vn;
                    conv[comp] += fo * (vf - vu);
                    tr[comp] += trc * (T(0.5) * (Gr[a][comp][c] + Gr[a][comp][nb]));
                }
            } else if (t == FT_WALL || t == FT_OUTLET) {
#pragma unroll
                for (int comp = 0; comp < DIM; ++comp) tr[comp] += sg * mu * Sa * Gr[a][comp][c];
            } else if (t == FT_INLET) {
                const T fo = sg * phic.a[a][f];
#pragma unroll
                for (int comp = 0; comp < DIM; ++comp) {
                    const T vin = comp == 0 ? vin0 : T(0);
                    lap[comp] += mul_S_div_half_h(g, gr, a, mu) * vin;
                    if (fo < T(0)) inflow[comp] += -fo * vin;
                    else conv[comp] += fo * (vin - vc[comp]);
                    tr[comp] += sg * mu * Sa * Gr[a][comp][c];
                }
            }
        }
    }
#pragma unroll
    for (int comp = 0; comp < DIM; ++comp) {
        T Hc = div_dt(gr, rho * vold.a[comp][c], dt);
        Hc += div_V(g, gr, lap[comp] + rho * (inflow[comp] - conv[comp]) + tr[comp]);
        hbya.a[comp][c] = rAc * Hc;
    }
}

// phi* of the face of direction A at face coordinates (i,j,k) (Section 2.2:
// interior faces (HbyA)_f S + (1/A)_f f_st S with arithmetic face means, the
// inlet U S, the outlet HbyA_L S, walls 0)
template <int A, typename T>
__device__ __forceinline__ T phistar_face(const GridD &g, const uint32_t *__restrict__ info, int i, int j, int k,
                                          const T *__restrict__ hbyaA, const T *__restrict__ rA,
                                          const T *__restrict__ fstA, T vinA) {
    int L, H;
    const int t = decode_face<A>(g, info, i, j, k, L, H);
    const T Sa = GA<T>::S(g, A);
    if (t == FT_INTERIOR)
        return T(0.5) * (hbyaA[L] + hbyaA[H]) * Sa + T(0.5) * (rA[L] + rA[H]) * fstA[flo(g, A, i, j, k)] * Sa;
    if (t == FT_INLET) return vinA * Sa;
    if (t == FT_OUTLET) return hbyaA[L] * Sa;
    return T(0);
}

// phi* of the faces of direction A around cell (i,j,k): its low face is
// stored (every face is the low face of one cell, or the high face of the
// last cell of a line), both enter the divergence
template <int A, typename T>
__device__ __forceinline__ void phistar_pair(const GridD &g, const uint32_t *__restrict__ info, int i, int j, int k,
                                             const T *__restrict__ hbyaA, const T *__restrict__ rA,
                                             const T *__restrict__ fstA, T vinA, T *__restrict__ phisA, T &div) {
    const T lo = phistar_face<A, T>(g, info, i, j, k, hbyaA, rA, fstA, vinA);
    const T hi = phistar_face<A, T>(g, info, i + (A == 0), j + (A == 1), k + (A == 2), hbyaA, rA, fstA, vinA);
    phisA[flo(g, A, i, j, k)] = lo;
    const int q = A == 0 ? i : (A == 1 ? j : k), n = A == 0 ? g.nx : (A == 1 ? g.ny : g.nz);
    if (q == n - 1) phisA[fhi(g, A, i, j, k)] = hi;
    div += -lo;
    div += hi;
}

// predicted fluxes phi* of every face and the pressure equation's right-hand
// side b = -div(phi*) in one cell kernel: each face value is computed by both
// of its cells with the same arithmetic, stored by the cell it is the low face
// of (or by the last cell of a line), and b sums the low and high faces of
// every direction in turn
template <int DIM, typename T>
__global__ void k_phistar_rhs(GridD g, const uint32_t *__restrict__ info, C3<T> hbya, const T *__restrict__ rA,
                              C3<T> fst, T vin0, P3<T> phis, double *__restrict__ b) {
    griddep_wait();
    CELL_IJK(g);
    if (!inside) return;
    T div = T(0);
    phistar_pair<0, T>(g, info, i, j, k, hbya.a[0], rA, fst.a[0], vin0, phis.a[0], div);
    phistar_pair<1, T>(g, info, i, j, k, hbya.a[1], rA, fst.a[1], T(0), phis.a[1], div);
    if constexpr (DIM == 3) phistar_pair<2, T>(g, info, i, j, k, hbya.a[2], rA, fst.a[2], T(0), phis.a[2], div);
    b[c] = (info[c] & INFO_FLUID) ? (double)(-div) : 0.0;
}

// corrected flux of the face of direction A at face coordinates (i,j,k):
// phi = phi* - c_f (q_H - q_L), the pressure difference taken in FP64 and
// rounded to T (q = 0 beyond the outlet face), unchanged on walls and at the
// inlet. dq: the rounded difference of this face when it is interior (the
// caller forms it once for the flux and the velocity correction).
template <int A, typename T>
__device__ __forceinline__ T corrected_face(const GridD &g, const uint32_t *__restrict__ info, int i, int j, int k,
                                            const T *__restrict__ phisA, const T *__restrict__ cfA,
                                            const double *__restrict__ q, T dq) {
    int L, H;
    const int t = decode_face<A>(g, info, i, j, k, L, H);
    const int f = flo(g, A, i, j, k);
    const T ps = phisA[f];
    if (t == FT_INTERIOR) return ps - cfA[f] * dq;
    if (t == FT_OUTLET) return ps - cfA[f] * (T)(0.0 - q[L]);
    return ps;
}

template <int A, typename T>
__device__ __forceinline__ void correct_pair(const GridD &g, const uint32_t *__restrict__ info, int i, int j, int k,
                                             const T *__restrict__ phisA, const T *__restrict__ cfA,
                                             const double *__restrict__ q, T dlo, T *__restrict__ phiA) {
    phiA[flo(g, A, i, j, k)] = corrected_face<A, T>(g, info, i, j, k, phisA, cfA, q, dlo);
    const int qq = A == 0 ? i : (A == 1 ? j : k), n = A == 0 ? g.nx : (A == 1 ? g.ny : g.nz);
    if (qq == n - 1)   // the domain's last face of the line is never interior
        phiA[fhi(g, A, i, j, k)] =
            corrected_face<A, T>(g, info, i + (A == 0), j + (A == 1), k + (A == 2), phisA, cfA, q, T(0));
}

// flux correction of every face and velocity correction v = HbyA + (1/A)
// reconstruct(face accelerations) (Section 2.2) in one cell kernel. Each
// interior face's pressure difference (T)(q_H - q_L) is formed once per cell
// that uses it: the low faces' by the cell, the high face in x taken from the
// next lane (the next cell of the row: a warp never spans two rows, block x
// extents being multiples of 32), the other high faces formed again. FP64
// instructions are scarce on this GPU, and this halves them.
template <int DIM, typename T>
__global__ void k_correct(GridD g, GR<T> gr, const uint32_t *__restrict__ info, C3<T> phis, C3<T> cf, const double *__restrict__ q,
                          P3<T> phi, C3<T> hbya, const T *__restrict__ rA, C3<T> fst, P3<T> v) {
    griddep_wait();
    CELL_IJK(g);
    const uint32_t inf = inside ? info[c] : 0u;
    const bool fluid = (inf & INFO_FLUID) != 0;
    const double qc = fluid ? q[c] : 0.0;
    T dlo[3] = {T(0), T(0), T(0)};
#pragma unroll
    for (int a = 0; a < DIM; ++a)
        if (fluid && ftype(inf, a, 0) == FT_INTERIOR) dlo[a] = (T)(qc - q[c - noff(g, a)]);
    const T dnext = __shfl_down_sync(0xffffffffu, dlo[0], 1);
    if (!inside) return;
    correct_pair<0, T>(g, info, i, j, k, phis.a[0], cf.a[0], q, dlo[0], phi.a[0]);
    correct_pair<1, T>(g, info, i, j, k, phis.a[1], cf.a[1], q, dlo[1], phi.a[1]);
    if constexpr (DIM == 3) correct_pair<2, T>(g, info, i, j, k, phis.a[2], cf.a[2], q, dlo[2], phi.a[2]);
    if (!fluid) {
#pragma unroll
        for (int a = 0; a < DIM; ++a) v.a[a][c] = T(0);
        return;
    }
    const bool next_in_warp = (threadIdx.x & 31) != 31;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        const int off = noff(g, a);
        T gs = T(0);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int t = ftype(inf, a, s);
            if (t == FT_INTERIOR) {
                const int f = s ? fhi(g, a, i, j, k) : flo(g, a, i, j, k);
                T dq;
                if (s == 0) dq = dlo[a];
                else if (a == 0 && next_in_warp) dq = dnext;
                else dq = (T)(q[c + off] - qc);
                gs += fst.a[a][f] - div_h(g, gr, a, dq);
            } else if (t == FT_OUTLET) {
                if constexpr (sizeof(T) == sizeof(double)) gs += div_half_h(g, gr, a, qc);
                else gs += -(T)(0.0 - qc) / (T(0.5) * GA<T>::h(g, a));
            }
        }
        v.a[a][c] = hbya.a[a][c] + rA[c] * T(0.5) * gs;
    }
}

// acc + w x: a product and a sum in FP32, fused in FP64 (half the FP64 instructions)
__device__ __forceinline__ float mg_madd(float w, float x, float acc) { return acc + w * x; }
__device__ __forceinline__ double mg_madd(double w, double x, double acc) { return fma(w, x, acc); }

// The FP64 operator row, sum over the faces of w_f (q_c - q_nb) (interior)
// and w_f q_c (outlet), from FP64 copies of the coefficients and with
// explicit FMAs: FP64 instructions are scarce on GB300, and this takes two
// per face. The differences are formed first, so a converged residual keeps
// its accuracy when q carries a large common level.
template <int DIM>
__device__ __forceinline__ double poisson_row64(const GridD &g, uint32_t inf, int c, int i, int j, int k,
                                                C3<double> w64, const double *__restrict__ q) {
    const double qc = q[c];
    double acc = 0.0;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        const int off = noff(g, a);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int t = ftype(inf, a, s);
            const int f = s ? fhi(g, a, i, j, k) : flo(g, a, i, j, k);
            if (t == FT_INTERIOR) acc = fma(w64.a[a][f], qc - q[s ? c + off : c - off], acc);
            else if (t == FT_OUTLET) acc = fma(w64.a[a][f], qc, acc);
        }
    }
    return acc;
}

// scal[slot] = scale * sum of x
template <typename T>
__global__ void k_sum_to(int n, const T *__restrict__ x, double scale, double *__restrict__ part,
                         unsigned *__restrict__ ticket, double *__restrict__ scal, int slot) {
    griddep_wait();
    double acc = 0.0, dummy = 0.0;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) acc += (double)x[c];
    if (reduce_last(acc, dummy, 1, false, part, 0, ticket, gridDim.x) && block_leader()) scal[slot] = acc * scale;
}

// u_sum += v and max |v - vold|; the finishing block applies the early exit
// of Section 3.2: stop after sub-step k if k = N or the test value (E_k, or
// max |du_cr| / U) is below the tolerance
template <int DIM, typename T>
__global__ void k_relax_accum(int n, const uint32_t *__restrict__ info, C3<T> v, C3<T> vold, P3<double> usum,
                              double *__restrict__ part, unsigned *__restrict__ ticket, double *__restrict__ scal,
                              int *__restrict__ ctl, int mode, double tol, double invU, cudaGraphConditionalHandle h) {
    griddep_wait();
    T mt = T(0);
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) {
        if (!(info[c] & INFO_FLUID)) continue;
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            T x = v.a[a][c];
            usum.a[a][c] += (double)x;
            T d = x - vold.a[a][c];
            mt = d > mt ? d : (-d > mt ? -d : mt);
        }
    }
    double m = (double)mt, dummy = 0.0;
    if (reduce_last(m, dummy, 1, true, part, 0, ticket, gridDim.x) && block_leader()) {
        scal[S_DUMAX] = m;
        int k = ++ctl[C_K];
        double E = scal[S_E];
        double dU = m * invU;
        double test = mode == OSCAR_CONV_DU_MAX ? dU : E;
        if (mode == OSCAR_CONV_AREA) {   // relative change of the relaxation's energy in this sub-step
            const double a0 = scal[S_AREA0], a1 = scal[S_AREA1];
            test = fabs(a1 - a0) / (a0 > 0.0 ? a0 : 1.0);
            scal[S_AREA0] = a1;
        }
        scal[S_DU] = dU;
        scal[S_TEST] = test;
        bool bad = !isfinite(test) || ctl[C_NAN];
        if (bad) ctl[C_NAN] = 1;
        set_cond(ctl, h, !bad && k < ctl[C_N] && !(test < tol));
    }
}

// ---------------------------------------------------------------------------
// CG. The residual of the outer (FP64) system is r = b - M q with q and b in
// FP64; the Krylov vectors are of type V (double on the FP64 path, float on
// the mixed path). Dot products are accumulated per thread in V (a thread
// takes several cells) and across threads and blocks in compensated FP32 pairs or FP64.
// ---------------------------------------------------------------------------
// The kernel also starts the first V-cycle: z receives the colour-0 half
// sweep of the finest level from z = 0 (z = r / diagonal on colour 0, 0 on
// colour 1), and the Krylov vectors named in zero1 / zero2 (may be null) are
// cleared. r64 (may be null) receives r in FP64. With inv_nf > 0 it also
// forms the normalised residual of Section 3.2 for the relaxation's exit
// test: E = sum |b - Mq| / (sum |Mq - M qbar| + sum |b - M qbar| + 1e-20),
// qbar the mean of q over the fluid cells (scal[S_QSUM] inv_nf), M qbar
// nonzero only through the outlet coefficients.
template <int DIM, typename T, typename V>
__global__ void k_cg_init(GridD g, const uint32_t *__restrict__ info, C3<double> w64, const double *__restrict__ q,
                          const double *__restrict__ b, V *__restrict__ r, double *__restrict__ r64,
                          const V *__restrict__ idiag0, V *__restrict__ z, V *__restrict__ zero1,
                          V *__restrict__ zero2, double *__restrict__ part,
                          int stride, unsigned *__restrict__ ticket, int nb, double *__restrict__ scal,
                          int *__restrict__ ctl, double rtol, int mode, cudaGraphConditionalHandle h,
                          double inv_nf) {
    griddep_wait();
    const bool with_E = inv_nf > 0.0;
    const double qbar = with_E ? scal[S_QSUM] * inv_nf : 0.0;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};   // b.b, r.r, sum |b - Mq|, the normalisation
    ROW_LOOP(g) {
        ROW_CELL(g);
        if (i >= g.nx) continue;
        uint32_t inf = info[c];
        V rv = V(0);
        double rc = 0.0;
        if (inf & INFO_FLUID) {
            const double bc = b[c];
            const double Mq = poisson_row64<DIM>(g, inf, c, i, j, k, w64, q);
            rc = bc - Mq;
            rv = (V)rc;
            acc[0] = fma(bc, bc, acc[0]);
            acc[1] = fma(rc, rc, acc[1]);
            if (with_E) {
                const double Mqbar = ftype(inf, 0, 1) == FT_OUTLET ? qbar * w64.a[0][fhi(g, 0, i, j, k)] : 0.0;
                acc[2] += fabs(bc - Mq);
                acc[3] += fabs(Mq - Mqbar) + fabs(bc - Mqbar);
            }
        }
        r[c] = rv;
        if (r64) r64[c] = rc;
        z[c] = ((i + j + k) & 1) == 0 ? rv * idiag0[c] : V(0);
        if (zero1) zero1[c] = V(0);
        if (zero2) zero2[c] = V(0);
    }
    if (reduce_last4(acc, with_E ? 4 : 2, part, stride, ticket, nb) && block_leader()) {
        scal[S_BB] = acc[0];
        scal[S_RR] = acc[1];
        if (with_E) {
            scal[S_RES] = acc[2];
            scal[S_NRM] = acc[3];
            scal[S_E] = acc[2] / (acc[3] + 1e-20);
        }
        residual_control(scal, ctl, rtol, mode, h);
    }
}

// beta = (r.z) / (r.z)_old (0 on the first iteration) from the partials of
// r.z, rounded to V, in every thread of the block; the first block stores r.z
// and counts the iteration. What does not depend on the partials is loaded
// beside them and stored after the barrier, here and in the other consumers:
// one round of dependent loads less in each (four steps of 1024x128 mixed 5.23
// -> 5.17 ms; three of 128x32x32 FP64 13.0 -> 12.75 ms, k_cg_apply_dot's
// coefficients before its wait included).
template <typename V>
__device__ __forceinline__ V cg_beta(const double *rz_part, int nrz, double *scal, int *ctl) {
    __shared__ V beta_s;
    const double ro = scal[S_RZ0];
    const int it = ctl[C_IT], its = ctl[C_ITSUM];
    const double rz = dot_total<V>(rz_part, nrz);
    if (block_leader()) beta_s = (V)(ro != 0.0 ? rz / ro : 0.0);
    __syncthreads();
    if (block_leader() && BLOCK_ID() == 0) {
        scal[S_RZ1] = rz;
        ctl[C_IT] = it + 1;
        ctl[C_ITSUM] = its + 1;
    }
    return beta_s;
}
// alpha = (r.z) / (p.Ap); the first block keeps r.z for the next beta
template <typename V>
__device__ __forceinline__ V cg_alpha(const double *pap_part, int npap, double *scal) {
    __shared__ V alpha_s;
    const double rz = scal[S_RZ1];
    const double pap = dot_total<V>(pap_part, npap);
    if (block_leader()) alpha_s = (V)(rz / pap);
    __syncthreads();
    if (block_leader() && BLOCK_ID() == 0) scal[S_RZ0] = rz;
    return alpha_s;
}

// FP64 path: Ap = M p and p.Ap. As in k_cg_pz_apply no face types are read and
// the coefficients are loaded before the grid dependency wait.
template <int DIM, typename V>
__global__ void __launch_bounds__(256) k_cg_apply_dot(GridD g, C3<V> cf, const V *__restrict__ p, V *__restrict__ Ap,
                                                      double *__restrict__ part, int groups) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x, nrow = g.ny * g.nz;
    const int off[3] = {1, g.nx, g.nx * g.ny}, n[3] = {g.nx, g.ny, g.nz};
    V w[2 * DIM];
    int c, ijk[3];
    bool in;
    auto load_fixed = [&](int row) {
        in = i < g.nx && row < nrow;
        const int k = DIM == 3 ? row / g.ny : 0;
        ijk[0] = i;
        ijk[1] = row - k * g.ny;
        ijk[2] = k;
        c = i + g.nx * row;
        if (in) {
            const int f0 = c + row, f1 = c + g.nx * k;
            w[0] = cf.a[0][f0];
            w[1] = cf.a[0][f0 + 1];
            w[2] = cf.a[1][f1];
            w[3] = cf.a[1][f1 + g.nx];
            if (DIM == 3) {
                w[4] = cf.a[2][c];
                w[5] = cf.a[2][c + off[2]];
            }
        }
    };
    int grp = blockIdx.y;
    load_fixed(grp * blockDim.y + threadIdx.y);
    griddep_wait();
    typename DotAcc<V>::type acc;
    for (;;) {
        if (in) {
            const V pc = p[c];
            V pn[2 * DIM], y = V(0);
#pragma unroll
            for (int a = 0; a < DIM; ++a) {
                pn[2 * a] = ijk[a] > 0 ? p[c - off[a]] : V(0);
                pn[2 * a + 1] = ijk[a] < n[a] - 1 ? p[c + off[a]] : V(0);
            }
#pragma unroll
            for (int q = 0; q < 2 * DIM; ++q) y = mg_madd(w[q], pc - pn[q], y);   // by axis, low face first
            Ap[c] = y;
            acc.add(pc * y);
        }
        grp += gridDim.y;
        if (grp >= groups) break;
        load_fixed(grp * blockDim.y + threadIdx.y);
    }
    dot_store(acc, part);
}

// Mixed path: p = z + beta p and Ap = M z + beta Ap (the search direction
// update folded into the operator apply: M p = M z + beta M p_old, so every
// thread writes only its own cell), then p.Ap; beta = 0 starts afresh. Each
// thread takes RPT rows of a group (launch_groups), loaded together; the face
// coefficients, fixed during a solve, are loaded before the grid dependency
// wait for its first group, the vectors after it. Faces that do not belong to
// the operator (walls, the inlet, faces of solid cells) have zero
// coefficients and z is 0 beyond the outlet, so no face types are read: the
// kernel was bound by instruction issue (55 % of its peak) with them.
template <int DIM, typename T, typename V, int RPT>
__global__ void __launch_bounds__(256) k_cg_pz_apply(GridD g, C3<T> cf, const V *__restrict__ z,
                              V *__restrict__ p, V *__restrict__ Ap, const double *__restrict__ rz_part, int nrz,
                              double *__restrict__ part, int groups, double *__restrict__ scal, int *__restrict__ ctl) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int nrow = g.ny * g.nz, step = blockDim.y * RPT;
    const int off[3] = {1, g.nx, g.nx * g.ny};
    T w[RPT][2 * DIM];
    V zc[RPT], zn[RPT][2 * DIM], po[RPT], ao[RPT];
    int c[RPT], j[RPT], k[RPT];
    bool in[RPT];
    auto load_fixed = [&](int row0) {
#pragma unroll
        for (int u = 0; u < RPT; ++u) {
            const int row = row0 + u * blockDim.y;
            in[u] = i < g.nx && row < nrow;
            k[u] = DIM == 3 ? row / g.ny : 0;
            j[u] = row - k[u] * g.ny;
            c[u] = i + g.nx * row;
            if (in[u]) {
                const int f0 = c[u] + row, f1 = c[u] + g.nx * k[u];
                w[u][0] = cf.a[0][f0];
                w[u][1] = cf.a[0][f0 + 1];
                w[u][2] = cf.a[1][f1];
                w[u][3] = cf.a[1][f1 + g.nx];
                if (DIM == 3) {
                    w[u][4] = cf.a[2][c[u]];
                    w[u][5] = cf.a[2][c[u] + off[2]];
                }
            }
        }
    };
    auto load_vectors = [&]() {
#pragma unroll
        for (int u = 0; u < RPT; ++u)
            if (in[u]) {
                const int ijk[3] = {i, j[u], k[u]}, n[3] = {g.nx, g.ny, g.nz};
                zc[u] = z[c[u]];
                po[u] = p[c[u]];
                ao[u] = Ap[c[u]];
#pragma unroll
                for (int a = 0; a < DIM; ++a) {
                    zn[u][2 * a] = ijk[a] > 0 ? z[c[u] - off[a]] : V(0);
                    zn[u][2 * a + 1] = ijk[a] < n[a] - 1 ? z[c[u] + off[a]] : V(0);
                }
            }
    };
    int grp = blockIdx.y;
    load_fixed(grp * step + threadIdx.y);
    griddep_wait();
    load_vectors();
    const V be = cg_beta<V>(rz_part, nrz, scal, ctl);
    const bool fresh = be == V(0);
    typename DotAcc<V>::type acc;
    for (;;) {
        V accv = V(0);
#pragma unroll
        for (int u = 0; u < RPT; ++u) {
            if (!in[u]) continue;
            const V pn = fresh ? zc[u] : zc[u] + be * po[u];
            V y = V(0);   // by axis, low face first
#pragma unroll
            for (int q = 0; q < 2 * DIM; ++q) y += (V)w[u][q] * (zc[u] - zn[u][q]);
            const V an = fresh ? y : y + be * ao[u];
            p[c[u]] = pn;
            Ap[c[u]] = an;
            accv += pn * an;
        }
        acc.add(accv);
        grp += gridDim.y;
        if (grp >= groups) break;
        load_fixed(grp * step + threadIdx.y);
        load_vectors();
    }
    dot_store(acc, part);
}

// x += alpha p, r -= alpha Ap, z = the first colour-0 half sweep of the next
// V-cycle (as in k_cg_init), and r.r. RPT rows per thread and group
// (launch_groups), loaded together. xfresh: x starts from 0 in the first
// iteration (what was read is dropped), so it needs no clearing beforehand.
template <typename V, int RPT>
__global__ void __launch_bounds__(256) k_cg_update(GridD g, V *__restrict__ x, V *__restrict__ r, const V *__restrict__ p,
                            const V *__restrict__ Ap, const V *__restrict__ idiag0, V *__restrict__ z,
                            const double *__restrict__ pap_part, int npap, double *__restrict__ part, int groups,
                            double *__restrict__ scal, const int *__restrict__ ctl, int xfresh) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int nrow = g.ny * g.nz;
    V id[RPT], xo[RPT], ro[RPT], pc[RPT], ac[RPT];
    auto load_fixed = [&](int row0) {
#pragma unroll
        for (int u = 0; u < RPT; ++u) {
            const int row = row0 + u * blockDim.y;
            id[u] = (i < g.nx && row < nrow) ? idiag0[i + g.nx * row] : V(0);
        }
    };
    int grp = blockIdx.y;
    const int step = blockDim.y * RPT;
    load_fixed(grp * step + threadIdx.y);
    griddep_wait();
    // with xfresh, the first iteration of a solve (counted by the kernel before) starts x from 0
    const bool x0 = xfresh && ctl[C_IT] == 1;
    auto load_vectors = [&](int row0) {
#pragma unroll
        for (int u = 0; u < RPT; ++u) {
            const int row = row0 + u * blockDim.y;
            if (i < g.nx && row < nrow) {
                const int c = i + g.nx * row;
                xo[u] = x[c];
                ro[u] = r[c];
                pc[u] = p[c];
                ac[u] = Ap[c];
            }
        }
    };
    load_vectors(grp * step + threadIdx.y);
    const V al = cg_alpha<V>(pap_part, npap, scal);
    typename DotAcc<V>::type acc;
    for (;;) {
        V accv = V(0);
#pragma unroll
        for (int u = 0; u < RPT; ++u) {
            const int row = grp * step + threadIdx.y + u * blockDim.y;
            if (i >= g.nx || row >= nrow) continue;
            const int c = i + g.nx * row;
            const int k = row / g.ny, j = row - k * g.ny;
            x[c] = x0 ? al * pc[u] : xo[u] + al * pc[u];
            const V rc = ro[u] - al * ac[u];
            r[c] = rc;
            z[c] = ((i + j + k) & 1) == 0 ? rc * id[u] : V(0);
            accv += rc * rc;
        }
        acc.add(accv);
        grp += gridDim.y;
        if (grp >= groups) break;
        load_fixed(grp * step + threadIdx.y);
        load_vectors(grp * step + threadIdx.y);
    }
    dot_store(acc, part);
}

// FP64 path, one block: ||r|| from the partials of r.r against the target;
// decides whether the PCG loop continues
template <typename V>
__global__ void k_cg_check(const double *__restrict__ rr_part, int nrr, double *__restrict__ scal, int *__restrict__ ctl,
                           int maxit, cudaGraphConditionalHandle h) {
    griddep_wait();
    const double rr = dot_total<V>(rr_part, nrr);
    if (!block_leader()) return;
    scal[S_RR] = rr;
    const double rn = sqrt(rr);
    const bool bad = !isfinite(rn);
    if (bad) ctl[C_NAN] = 1;
    bool more = !bad && rn > scal[S_TARGET];
    if (more && ctl[C_IT] >= maxit) { ctl[C_NOTCONV] = 1; more = false; }
    set_cond(ctl, h, more);
}

// r.z, cell by cell (when the whole V-cycle ran in the cluster)
template <typename V>
__global__ void k_cg_dot_rz(int n, const V *__restrict__ x, const V *__restrict__ y, double *__restrict__ part) {
    griddep_wait();
    typename DotAcc<V>::type acc;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += gridDim.x * blockDim.x) acc.add(x[c] * y[c]);
    dot_store(acc, part);
}

// p = z + beta p
template <typename V>
__global__ void k_cg_pupdate(int n, const V *__restrict__ z, V *__restrict__ p, const double *__restrict__ rz_part, int nrz,
                             double *__restrict__ scal, int *__restrict__ ctl) {
    griddep_wait();
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    V zc = V(0), pc = V(0);   // of the first cell, beside the partials
    if (c < n) {
        zc = z[c];
        pc = p[c];
    }
    const V be = cg_beta<V>(rz_part, nrz, scal, ctl);
    if (c < n) p[c] = zc + be * pc;
    while ((c += gridDim.x * blockDim.x) < n) p[c] = z[c] + be * p[c];
}

// Error-free products (FMA) for the compensated operator below.
__device__ __forceinline__ void two_prod(float a, float b, float &p, float &e) {
    p = a * b;
    e = fmaf(a, b, -p);
}

// (M e)_c of an FP32 vector with FP32 coefficients as an unevaluated pair of
// floats s + cc: each face difference (TwoSum) and product (TwoProduct) is
// formed without rounding error and the terms are summed with TwoSum, so the
// pair matches the exact row value to about 2^-46 of the sum of the term
// magnitudes -- FP64-grade, with FP32 instructions only. Same faces as
// poisson_row64.
template <int DIM>
__device__ __forceinline__ void poisson_row_comp(const GridD &g, uint32_t inf, int c, int i, int j, int k,
                                                 C3<float> cf, const float *__restrict__ e, float &s, float &cc) {
    const float ec = e[c];
    s = 0.f;
    cc = 0.f;
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        const int off = noff(g, a);
#pragma unroll
        for (int sd = 0; sd < 2; ++sd) {
            const int t = ftype(inf, a, sd);
            if (t != FT_INTERIOR && t != FT_OUTLET) continue;
            const float w = cf.a[a][sd ? fhi(g, a, i, j, k) : flo(g, a, i, j, k)];
            float p, pe, lo = 0.f;
            if (t == FT_INTERIOR) {
                float dh;
                two_sum(ec, -e[sd ? c + off : c - off], dh, lo);
                two_prod(w, dh, p, pe);
                pe += w * lo;
            } else {
                two_prod(w, ec, p, pe);
            }
            float sn, se;
            two_sum(s, p, sn, se);
            s = sn;
            cc += se + pe;
        }
    }
}

// Mixed path, the last kernel of an iteration: every block forms ||r|| from
// the partials of r.r (the same value everywhere) and decides whether the FP32
// iteration goes on; if so, that is all. Otherwise the defect-correction trip
// ends: q += e in FP64, and the FP64 residual updated recursively, r64 -= M e,
// with M e from the compensated apply above (so r64 stays b - M q to FP64
// accuracy, without re-evaluating the operator on q in FP64); then
// r = (float) r64, z = the first colour-0 half sweep of the next V-cycle,
// ||r||^2, and the loop decision of residual_control(mode 2). With the trip's
// end inside the iteration a solve is one loop: a loop of iterations inside
// one of trips costs 5 us to enter and to leave per trip, more than the
// 1.5 us of the iterations that only check. The values the decision reads are
// written by the last block to finish at the earliest.
template <int DIM>
__global__ void __launch_bounds__(1024) k_cg_refine(GridD g, const uint32_t *__restrict__ info, C3<float> cf, const float *__restrict__ e,
                            double *__restrict__ q, double *__restrict__ r64, float *__restrict__ r,
                            const float *__restrict__ idiag0, float *__restrict__ z, const double *__restrict__ rr_part,
                            int nrr, double *__restrict__ part, int stride, unsigned *__restrict__ ticket, int nb,
                            double *__restrict__ scal, int *__restrict__ ctl, double rtol, int maxit,
                            cudaGraphConditionalHandle h) {
    griddep_wait();
    __shared__ int more_s;
    {
        const double target = scal[S_ITARGET];
        const int it = ctl[C_IT];
        const double rr = dot_total<float>(rr_part, nrr);
        if (block_leader()) {
            const double rn = sqrt(rr);
            const bool bad = !isfinite(rn);
            bool more = !bad && rn > target;
            const bool capped = more && it >= maxit;
            if (capped) more = false;
            if (BLOCK_ID() == 0) {
                if (bad) ctl[C_NAN] = 1;
                if (capped) ctl[C_NOTCONV] = 1;
                if (more) set_cond(ctl, h, true);
            }
            more_s = more;
        }
        __syncthreads();
        if (more_s) return;
    }
    double rr = 0.0, dummy = 0.0;
    ROW_LOOP(g) {
        ROW_CELL(g);
        if (i >= g.nx) continue;
        const uint32_t inf = info[c];
        float rv = 0.f;
        if (inf & INFO_FLUID) {
            float s, cc;
            poisson_row_comp<DIM>(g, inf, c, i, j, k, cf, e, s, cc);
            q[c] += (double)e[c];
            const double rn = r64[c] - ((double)s + (double)cc);
            r64[c] = rn;
            rv = (float)rn;
            rr = fma(rn, rn, rr);
        }
        r[c] = rv;
        z[c] = ((i + j + k) & 1) == 0 ? rv * idiag0[c] : 0.f;
    }
    if (reduce_last(rr, dummy, 1, false, part, stride, ticket, nb) && block_leader()) {
        scal[S_RR] = rr;
        residual_control(scal, ctl, rtol, 2, h);
    }
}


// ---------------------------------------------------------------------------
// geometric multigrid (preconditioner): piecewise-constant transfers, coarse
// operators from summed fine face coefficients (x 1/2 across a coarsened
// direction), red-black Gauss-Seidel smoothing
// ---------------------------------------------------------------------------
template <typename M> struct MG3 { const M *a[3]; };

// neighbour coefficients of a row (zero across the domain boundary); the
// per-level kernels load them, and the other operands that stay fixed during
// a solve, before griddep_wait, so that only the operands written by the
// preceding kernel are loaded after it (one round of dependent loads). The
// coefficient arrays and (inverse) diagonals are written by the set-up of a
// PISO corrector, never by the kernel that directly precedes a reader.
template <int DIM, typename M>
__device__ __forceinline__ void mg_row_coeffs(const GridD &g, MG3<M> cc, int i, int j, int k, M *w) {
    const int ijk[3] = {i, j, k}, n[3] = {g.nx, g.ny, g.nz};
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        w[2 * a] = ijk[a] > 0 ? cc.a[a][flo(g, a, i, j, k)] : M(0);
        w[2 * a + 1] = ijk[a] < n[a] - 1 ? cc.a[a][fhi(g, a, i, j, k)] : M(0);
    }
}
// b + the sum of the neighbour terms of a row
template <int DIM, typename M, typename F>
__device__ __forceinline__ M mg_row_sum(const GridD &g, const M *w, M b, int i, int j, int k, F x) {
    const int ijk[3] = {i, j, k}, n[3] = {g.nx, g.ny, g.nz};
    M acc = sizeof(M) == sizeof(double) ? b : M(0);
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
        if (ijk[a] > 0) acc = mg_madd(w[2 * a], x(a, 0), acc);
        if (ijk[a] < n[a] - 1) acc = mg_madd(w[2 * a + 1], x(a, 1), acc);
    }
    return sizeof(M) == sizeof(double) ? acc : b + acc;
}
template <int DIM, typename M>
__device__ __forceinline__ M mg_row_sum(const GridD &g, const M *w, M b, const M *x, int cell, int i, int j, int k) {
    return mg_row_sum<DIM, M>(g, w, b, i, j, k, [&](int a, int s) { return x[s ? cell + noff(g, a) : cell - noff(g, a)]; });
}
// b - M x of a row with diagonal dg
template <int DIM>
__device__ __forceinline__ float mg_residual(const GridD &g, const float *w, float dg, float b, const float *x, int cell, int i,
                                             int j, int k) {
    return b - (dg * x[cell] - mg_row_sum<DIM, float>(g, w, 0.f, x, cell, i, j, k));
}
template <int DIM>
__device__ __forceinline__ double mg_residual(const GridD &g, const double *w, double dg, double b, const double *x, int cell,
                                              int i, int j, int k) {
    return fma(-dg, x[cell], mg_row_sum<DIM, double>(g, w, b, x, cell, i, j, k));
}

// one colour of a red-black Gauss-Seidel sweep; thread ti handles the cell
// i = 2 ti + ((j + k + colour) & 1) of its row, so no thread idles. idiag is
// 1 / diagonal on fluid cells and 0 elsewhere, so solid cells keep x = 0.
// PRO: the first post-smoothing half sweep with the prolongation folded in:
// every neighbour value is read as x + xc(parent), which is what the
// piecewise-constant prolongation would have stored (faces to solid cells
// have zero coefficients, so their values do not matter). The other colour
// is never read before the next half sweep overwrites it, so the prolonged
// field itself is not stored.
// DG: the inverse diagonal formed from the row's coefficients, with the
// operations of k_mg_diag, instead of read: one of the seven values per cell
// that a 3D half sweep moves (15.9 us for 117 MB at 256x128x128, at the rate of
// the HBM). On levels that stay in L2 the division costs more than the load.
template <int DIM, typename M, bool PRO, bool DG>
__global__ void k_mg_rbgs(GridD g, MG3<M> cc, const M *__restrict__ idiag, M *__restrict__ x,
                          const M *__restrict__ b, int colour, GridD gc, int s0, int s1, int s2,
                          const M *__restrict__ xc) {
    const int ti = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z;
    const int i = 2 * ti + ((j + k + colour) & 1);
    const bool ok = i < g.nx && j < g.ny;
    const int cell = i + g.nx * (j + g.ny * k);
    M w[2 * DIM], id = M(0);
    if (ok) {
        if constexpr (DG) {
            const int ijk[3] = {i, j, k}, n[3] = {g.nx, g.ny, g.nz};
            M d = M(0);   // as k_mg_diag
#pragma unroll
            for (int a = 0; a < DIM; ++a) {
                const M lo = cc.a[a][flo(g, a, i, j, k)], hi = cc.a[a][fhi(g, a, i, j, k)];
                d += lo + hi;
                w[2 * a] = ijk[a] > 0 ? lo : M(0);   // as mg_row_coeffs
                w[2 * a + 1] = ijk[a] < n[a] - 1 ? hi : M(0);
            }
            id = d > M(0) ? M(1) / d : M(0);
        } else {
            mg_row_coeffs<DIM, M>(g, cc, i, j, k, w);
            id = idiag[cell];
        }
    }
    griddep_wait();
    if (!ok) return;
    const M bc = b[cell];
    M t;
    if constexpr (PRO) {
        const int sh[3] = {s0, s1, s2}, ijk[3] = {i, j, k};
        t = mg_row_sum<DIM, M>(g, w, bc, i, j, k, [&](int a, int s) {
            int pp[3] = {i >> s0, j >> s1, k >> s2};
            pp[a] = (ijk[a] + (s ? 1 : -1)) >> sh[a];
            return x[s ? cell + noff(g, a) : cell - noff(g, a)] + xc[pp[0] + gc.nx * (pp[1] + gc.ny * pp[2])];
        });
    } else {
        t = mg_row_sum<DIM, M>(g, w, bc, x, cell, i, j, k);
    }
    x[cell] = t * id;
}

// The last half sweep of the finest level (colour 0) fused with r.z: the
// thread of colour cell i also takes its row partner i ^ 1 (colour 1, final
// already), so every cell is counted once. A thread takes RPT rows of a group
// (launch_groups over the colour's cells), loaded together.
template <int DIM, typename M, int RPT>
__global__ void __launch_bounds__(256) k_mg_rbgs_dot(GridD g, MG3<M> cc, const M *__restrict__ idiag, M *__restrict__ x,
                              const M *__restrict__ b, int colour, int groups, double *__restrict__ part) {
    const int ti = blockIdx.x * blockDim.x + threadIdx.x;
    const int nrow = g.ny * g.nz, step = blockDim.y * RPT;
    int grp = blockIdx.y;
    M w[RPT][2 * DIM], id[RPT];
    int row[RPT], j[RPT], k[RPT], i[RPT];
    bool ok[RPT];
    auto load_fixed = [&]() {
#pragma unroll
        for (int u = 0; u < RPT; ++u) {
            row[u] = grp * step + threadIdx.y + u * blockDim.y;
            k[u] = DIM == 3 ? row[u] / g.ny : 0;
            j[u] = row[u] - k[u] * g.ny;
            i[u] = 2 * ti + ((j[u] + k[u] + colour) & 1);
            ok[u] = i[u] < g.nx && row[u] < nrow;
            if (ok[u]) {
                mg_row_coeffs<DIM, M>(g, cc, i[u], j[u], k[u], w[u]);
                id[u] = idiag[i[u] + g.nx * row[u]];
            }
        }
    };
    load_fixed();
    griddep_wait();
    typename DotAcc<M>::type sum;
    for (;;) {
        M bc[RPT], xn[RPT], bp[RPT], xp[RPT];
#pragma unroll
        for (int u = 0; u < RPT; ++u) {
            const int cell = i[u] + g.nx * row[u], ip = i[u] ^ 1, cellp = ip + g.nx * row[u];
            const bool okp = ip < g.nx && row[u] < nrow;
            bp[u] = okp ? b[cellp] : M(0);
            xp[u] = okp ? x[cellp] : M(0);
            if (ok[u]) {
                bc[u] = b[cell];
                xn[u] = mg_row_sum<DIM, M>(g, w[u], bc[u], x, cell, i[u], j[u], k[u]) * id[u];
            }
        }
#pragma unroll
        for (int u = 0; u < RPT; ++u) {
            M acc = M(0);
            if (ok[u]) {
                x[i[u] + g.nx * row[u]] = xn[u];
                acc = bc[u] * xn[u];
            }
            acc += bp[u] * xp[u];
            sum.add(acc);
        }
        grp += gridDim.y;
        if (grp >= groups) break;
        load_fixed();
    }
    dot_store(sum, part);
}

// coarse b = sum over children of the fine residual b - M x (0 on solid cells,
// which have no coefficients and b = 0). With first set,
// the coarse x receives the first colour-0 half sweep from x = 0
// (x = b / diagonal on colour 0, 0 on colour 1), else x = 0. One thread per
// fine cell: a block covers a tile of whole coarse cells (even extents,
// kRRTile), puts the residuals of its fine cells in shared memory, and one
// thread per coarse cell of the tile sums the children in the order x fastest.
// On the small middle levels this spreads a launch over 8x the threads of a
// thread-per-coarse-cell kernel, whose chain of child loads set its latency.
template <int DIM> struct RRTile {
    static constexpr int X = 32, Y = DIM == 3 ? 4 : 8, Z = DIM == 3 ? 2 : 1;
};
template <int DIM, typename M, int RX, int RY, int RZ>
__global__ void __launch_bounds__(256) k_mg_resid_restrict(GridD gf, GridD gc, MG3<M> cc,
                                                           const M *__restrict__ diag,
                                                           const M *__restrict__ x, const M *__restrict__ b,
                                                           M *__restrict__ bc, M *__restrict__ xc,
                                                           const M *__restrict__ idc, int first) {
    constexpr int TX = RRTile<DIM>::X, TY = RRTile<DIM>::Y, TZ = RRTile<DIM>::Z;
    constexpr int CX = TX / RX, CY = TY / RY, CZ = TZ / RZ, NC = CX * CY * CZ;
    __shared__ M res[TX * TY * TZ];
    const int t = threadIdx.x + TX * (threadIdx.y + TY * threadIdx.z);
    const int i = blockIdx.x * TX + threadIdx.x, j = blockIdx.y * TY + threadIdx.y, k = blockIdx.z * TZ + threadIdx.z;
    const bool in = i < gf.nx && j < gf.ny && k < gf.nz;
    const int cell = i + gf.nx * (j + gf.ny * k);
    M w[2 * DIM], dg = M(0);
    if (in) {
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
            w[2 * a] = cc.a[a][flo(gf, a, i, j, k)];
            w[2 * a + 1] = cc.a[a][fhi(gf, a, i, j, k)];
            // FP32: the diagonal as k_mg_diag and k_mg_level_operator form it,
            // 4 bytes per cell less to read; FP64 is bound by its additions
            if (sizeof(M) == sizeof(float)) dg += w[2 * a] + w[2 * a + 1];
        }
        if (sizeof(M) == sizeof(double)) dg = diag[cell];
    }
    int ic = 0, jc = 0, kc = 0;
    bool cin = false;
    M idq = M(0);
    if (t < NC) {
        ic = blockIdx.x * CX + t % CX;
        jc = blockIdx.y * CY + (t / CX) % CY;
        kc = blockIdx.z * CZ + t / (CX * CY);
        cin = ic < gc.nx && jc < gc.ny && kc < gc.nz;
        if (cin && first) idq = idc[ic + gc.nx * (jc + gc.ny * kc)];
    }
    griddep_wait();
    M rv = M(0);
    if (in) {
        rv = mg_residual<DIM>(gf, w, dg, b[cell], x, cell, i, j, k);
    }
    res[t] = rv;
    __syncthreads();
    if (!cin) return;
    M acc = M(0);
#pragma unroll
    for (int qz = 0; qz < RZ; ++qz)
#pragma unroll
        for (int qy = 0; qy < RY; ++qy)
#pragma unroll
            for (int qx = 0; qx < RX; ++qx) {
                const int ii = ic * RX + qx, jj = jc * RY + qy, kk = kc * RZ + qz;
                if (ii >= gf.nx || jj >= gf.ny || kk >= gf.nz) continue;
                acc += res[(ii - (int)blockIdx.x * TX) + TX * ((jj - (int)blockIdx.y * TY) + TY * (kk - (int)blockIdx.z * TZ))];
            }
    const int cq = ic + gc.nx * (jc + gc.ny * kc);
    bc[cq] = acc;
    xc[cq] = (first && ((ic + jc + kc) & 1) == 0) ? acc * idq : M(0);
}

static __global__ void k_mg_fluid_coarsen(GridD gf, GridD gc, int rx, int ry, int rz, const uint8_t *__restrict__ ff,
                                          uint8_t *__restrict__ fc) {
    griddep_wait();
    CELL_IJK(gc);
    if (!inside) return;
    uint8_t any = 0;
    for (int oz = 0; oz < rz; ++oz)
        for (int oy = 0; oy < ry; ++oy)
            for (int ox = 0; ox < rx; ++ox) {
                int ii = i * rx + ox, jj = j * ry + oy, kk = k * rz + oz;
                if (ii < gf.nx && jj < gf.ny && kk < gf.nz && ff[ii + gf.nx * (jj + gf.ny * kk)]) any = 1;
            }
    fc[c] = any;
}

// coarse face coefficient of direction A at face coordinates (i,j,k) of the
// coarse grid: sum of the fine faces covering it, halved across a coarsened
// direction
template <int A, typename M>
__device__ __forceinline__ M coarse_face(const GridD &gf, int i, int j, int k, int rx, int ry, int rz,
                                         const M *__restrict__ cfine) {
    const int rr[3] = {rx, ry, rz};
    const int nfn[3] = {gf.nx, gf.ny, gf.nz};
    const int base[3] = {i, j, k};
    int lo[3], cnt[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        if (b == A) {
            lo[b] = rr[b] == 2 ? min(2 * base[b], nfn[b]) : base[b];
            cnt[b] = 1;
        } else {
            lo[b] = base[b] * rr[b];
            cnt[b] = min(rr[b], nfn[b] - lo[b]);
        }
    }
    M acc = M(0);
    for (int oz = 0; oz < cnt[2]; ++oz)
        for (int oy = 0; oy < cnt[1]; ++oy)
            for (int ox = 0; ox < cnt[0]; ++ox) acc += cfine[flo(gf, A, lo[0] + ox, lo[1] + oy, lo[2] + oz)];
    return rr[A] == 2 ? M(0.5) * acc : acc;
}

// A coarse level's operator in one cell kernel: the face coefficients from
// the finer level's (coarse_face; each face stored by the cell it is the low
// face of, or by the last cell of its line) and the diagonal with its
// reciprocal, as k_mg_diag forms them from the stored faces. The high faces
// a cell needs for its diagonal are formed again with the same arithmetic,
// so the values are those of a face pass followed by a diagonal pass.
template <int A, typename M>
__device__ __forceinline__ M coarse_face_pair(const GridD &gf, const GridD &gc, int i, int j, int k, int rx, int ry,
                                              int rz, const M *__restrict__ cfine, M *__restrict__ ccoarse) {
    const M lo = coarse_face<A, M>(gf, i, j, k, rx, ry, rz, cfine);
    const M hi = coarse_face<A, M>(gf, i + (A == 0), j + (A == 1), k + (A == 2), rx, ry, rz, cfine);
    ccoarse[flo(gc, A, i, j, k)] = lo;
    const int q = A == 0 ? i : (A == 1 ? j : k), n = A == 0 ? gc.nx : (A == 1 ? gc.ny : gc.nz);
    if (q == n - 1) ccoarse[fhi(gc, A, i, j, k)] = hi;
    return lo + hi;
}
template <int DIM, typename M>
__global__ void k_mg_level_operator(GridD gf, GridD gc, int rx, int ry, int rz, MG3<M> cfine, P3<M> ccoarse,
                                    const uint8_t *__restrict__ fluid, M *__restrict__ diag, M *__restrict__ idiag) {
    griddep_wait();
    CELL_IJK(gc);
    if (!inside) return;
    M acc = M(0);
    acc += coarse_face_pair<0, M>(gf, gc, i, j, k, rx, ry, rz, cfine.a[0], ccoarse.a[0]);
    acc += coarse_face_pair<1, M>(gf, gc, i, j, k, rx, ry, rz, cfine.a[1], ccoarse.a[1]);
    if constexpr (DIM == 3) acc += coarse_face_pair<2, M>(gf, gc, i, j, k, rx, ry, rz, cfine.a[2], ccoarse.a[2]);
    if (!fluid[c]) { diag[c] = M(0); idiag[c] = M(0); return; }
    diag[c] = acc;
    idiag[c] = acc > M(0) ? M(1) / acc : M(0);
}

// diagonal (sum of the face coefficients) and its reciprocal (0 on solid cells
// and on fluid cells without coefficients)
template <int DIM, typename M>
__global__ void k_mg_diag(GridD g, const uint8_t *__restrict__ fluid, MG3<M> cc, M *__restrict__ diag,
                          M *__restrict__ idiag) {
    griddep_wait();
    CELL_IJK(g);
    if (!inside) return;
    if (!fluid[c]) { diag[c] = M(0); idiag[c] = M(0); return; }
    M acc = M(0);
#pragma unroll
    for (int a = 0; a < DIM; ++a) acc += cc.a[a][flo(g, a, i, j, k)] + cc.a[a][fhi(g, a, i, j, k)];
    diag[c] = acc;
    idiag[c] = acc > M(0) ? M(1) / acc : M(0);
}

// idx -> (a, b, c) with idx = a + n0 * (b + n1 * c), without integer
// division (float reciprocals, corrected by one step; exact below 2^22)
__device__ __forceinline__ void split3(int idx, int n0, float rn0, int n1, float rn1, int &a, int &b, int &c) {
    int r = (int)(((float)idx + 0.5f) * rn0);
    a = idx - r * n0;
    if (a < 0) { --r; a += n0; } else if (a >= n0) { ++r; a -= n0; }
    c = (int)(((float)r + 0.5f) * rn1);
    b = r - c * n1;
    if (b < 0) { --c; b += n1; } else if (b >= n1) { ++c; b -= n1; }
}

}  // namespace oscar
