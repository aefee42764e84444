"""The thread-block-cluster kernels, and other size-dependent forms, against the paths they stand in for.

A pressure solve of a small 2D grid runs in one cluster, and the coarse levels
of larger grids in another; with cta_global=0 the same levels are worked by
per-level kernels and a cluster of one CTA. Mixed path: the same operations on
the same operands, so the fields are bitwise equal. FP64 path: other orders of
summation; with the solves converged to 1e-13 the fields agree to 1e-9 of
their largest value.
"""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2105_10576_gb300 import inputs
from paper_2105_10576_gb300 import oscar as ox

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def _sim(shape, prec, rtol, seed, solid_frac=0.15, **sched):
    nx, ny, nz = shape
    c = inputs.random_small_case(seed, nx, ny, nz=nz, dim=3 if nz > 1 else 2, solid_frac=solid_frac)
    p = dict(c.params, precision=prec, cg_rtol=rtol, conv_mode=inputs.CONV_PRES_RESID, conv_tol=0.0)
    g = ox.Oscar(p, c.solid, c.alpha0)
    g.set_schedule(sched)
    dt_cfl, dt_b, dt_vd, N = ox.oscar_timesteps(p, 0.02)
    return g, p, dt_vd, N


# one, two and three slab columns per CTA, ragged slabs, the line between 8 and
# 16 CTAs (2048 cells) and between 256 and 512 threads (8192), the largest grid
# solved whole (16384) and the first beyond it, larger grids' levels in 8 CTAs;
# in 3D slabs that end inside the grid (every level coarsens all axes by 2 here)
SHAPES = [(16, 8, 1), (37, 19, 1), (64, 32, 1), (129, 16, 1), (65, 33, 1), (256, 32, 1), (241, 35, 1), (257, 63, 1),
          (256, 64, 1), (257, 64, 1), (512, 128, 1), (513, 128, 1), (33, 9, 21), (48, 40, 7), (50, 27, 26), (70, 12, 12)]


@pytest.mark.parametrize("prec", [inputs.PREC_MIXED, inputs.PREC_FP64])
@pytest.mark.parametrize("sweeps", [dict(), dict(mg_nu=1, mg_nu_mid=3, mg_nu_cta=1, cta_cells=256)])
@pytest.mark.parametrize("shape", SHAPES)
def test_cluster_is_the_launched_path(shape, sweeps, prec):
    mixed = prec == inputs.PREC_MIXED
    out = []
    for flag in (1, 0):
        g, p, dt_vd, N = _sim(shape, prec, 1e-8 if mixed else 1e-13, 5 + shape[0], cta_global=flag, **sweeps)
        g.drag_step(dt_vd)
        g.relax(dt_vd / N, 2)
        out.append([g.field(w) for w in (ox.FIELD_ALPHA, ox.FIELD_P, ox.FIELD_U, ox.FIELD_U + 1, ox.FIELD_PHI_VD)])
        g.close()
    for x, y in zip(*out):
        if mixed:
            assert np.array_equal(x, y)
        else:
            assert np.abs(x - y).max() <= 1e-9 * np.abs(y).max()


# grids of one level: the V-cycle is the explicit inverse itself, so PCG needs
# one iteration (FP64; one more for rounding), or with the FP32 inverse, off by
# at most 1e-2 at the grids' density contrast, three per defect-correction trip
# of 1e-4, three trips to 1e-9. Bands of 1 to 25, an even and an odd middle,
# grids shorter than their band, the full 128 cells.
@pytest.mark.parametrize("prec,most", [(inputs.PREC_FP64, 2), (inputs.PREC_MIXED, 9)])
@pytest.mark.parametrize("shape", [(32, 4, 1), (16, 8, 1), (11, 11, 1), (19, 4, 1), (9, 3, 1), (4, 3, 1), (4, 32, 1),
                                   (5, 5, 5), (4, 5, 6), (32, 2, 2), (2, 3, 21), (8, 4, 4), (3, 3, 3)])
def test_coarsest_inverse(shape, prec, most):
    g, p, dt_vd, N = _sim(shape, prec, 1e-9, 3, coarse_refresh=1)
    g.drag_step(dt_vd)
    assert g.stats()["cg_iters_total"] <= most * p["n_piso"]
    assert np.isfinite(g.field(ox.FIELD_P)).all()
    g.close()


# the smallest ragged grids whose finest half sweeps form the inverse diagonal
# from the coefficients: a mixed step against the FP64 path, which reads it.
# alpha as in the other mixed tests; a wrong diagonal would cost iterations
# (the FP32 trips restart the iteration: at most twice the FP64 path's)
@pytest.mark.parametrize("shape", [(255, 131, 101), (2051, 1951, 1)])
def test_diagonal_from_coefficients(shape):
    alpha, its = [], []
    for prec in (inputs.PREC_MIXED, inputs.PREC_FP64):
        g, p, dt_vd, N = _sim(shape, prec, 1e-8, 7, solid_frac=0.02)
        g.drag_step(dt_vd)
        alpha.append(g.field(ox.FIELD_ALPHA))
        its.append(g.stats()["cg_iters_total"])
        g.close()
    assert np.abs(alpha[0] - alpha[1]).max() <= 1e-5
    assert its[0] <= 2 * its[1]


def _clusters(g, dt_vd):
    """CTAs of every cluster kernel that a drag step launches, by kernel name."""
    g.profile(True)
    g.drag_step(dt_vd)
    g.profile(False)
    rows = [(name.split("<")[0].split(" ")[-1].split("::")[-1], grid) for name, grid, _, _ in g.profile_read()]
    return {name: grid for name, grid in rows if "_cluster" in name}


# the V-cycle's cluster: as many CTAs as the coarsest level has columns, at most
# 8 (instances stepped together wait for wider ones)
@pytest.mark.parametrize("shape,ctas", [((512, 128, 1), 8), ((256, 32, 32), 8), ((64, 64, 64), 4), ((24, 40, 40), 2)])
@pytest.mark.parametrize("prec", [inputs.PREC_MIXED, inputs.PREC_FP64])
def test_vcycle_cluster_width(shape, ctas, prec):
    g, p, dt_vd, N = _sim(shape, prec, 1e-8, 11, solid_frac=0.05)
    assert _clusters(g, dt_vd) == {"k_mg_cluster": ctas}
    g.set_schedule(dict(cta_global=0))
    assert _clusters(g, dt_vd) == {"k_mg_cluster": 1}
    g.close()


# the levels above 1024 cells that the cluster takes: those of which a CTA works
# at most 2048 rows (levels counted from the finest, 0; -1: none)
@pytest.mark.parametrize("shape,level", [((512, 128, 1), 2), ((256, 32, 32), 2), ((64, 512, 1), 2), ((16, 1024, 1), -1),
                                         ((64, 64, 64), -1), ((32, 32, 32), -1)])
def test_vcycle_cluster_levels(shape, level):
    g, p, dt_vd, N = _sim(shape, inputs.PREC_MIXED, 1e-8, 11, solid_frac=0.05)
    assert g.stats()["mg_cta_global_level"] == level
    g.close()


# a schedule whose images need more than the default one's: room is made for
# them, and the steps are those of the launched path; back to the default
@pytest.mark.parametrize("shape", [(256, 32, 1), (257, 65, 1), (70, 24, 24)])
def test_schedule_with_larger_images(shape):
    wide = dict(mg_nu=4, mg_nu_mid=4, mg_nu_cta=6)
    out, held = [], []
    for flag in (1, 0):
        g, p, dt_vd, N = _sim(shape, inputs.PREC_MIXED, 1e-8, 23, cta_global=flag)
        assert flag == 0 or g.stats()["device_bytes"] == ox.oscar_footprint(p)
        for sched in (wide, dict(mg_nu=2, mg_nu_mid=2, mg_nu_cta=2), wide):
            g.set_schedule(sched)
            g.drag_step(dt_vd)
        held.append(g.stats()["device_bytes"] - ox.oscar_footprint(p))
        out.append([g.field(w) for w in (ox.FIELD_ALPHA, ox.FIELD_P, ox.FIELD_U)])
        g.close()
    assert 0 < held[0] < 2.1e6 and held[1] == 0
    for x, y in zip(*out):
        assert np.array_equal(x, y)


def _preload(tmp_path, source):
    from paper_2105_10576_gb300 import build
    src, lib = tmp_path / "fake.c", tmp_path / "fake.so"
    src.write_text(source)
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc()))), "include")
    subprocess.run(["gcc", "-shared", "-fPIC", "-I" + inc, "-o", str(lib), str(src), "-ldl"], check=True)
    return str(lib)


FAKE_OCCUPANCY = r"""
#include <cuda_runtime.h>
#include <stdlib.h>
/* a device on which clusters of more than FAKE_CLUSTER CTAs cannot be placed */
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *f, const cudaLaunchConfig_t *cfg) {
    unsigned nc = 1;
    for (unsigned q = 0; q < cfg->numAttrs; ++q)
        if (cfg->attrs[q].id == cudaLaunchAttributeClusterDimension) nc = cfg->attrs[q].val.clusterDim.x;
    *n = nc <= (unsigned)atoi(getenv("FAKE_CLUSTER"));
    return cudaSuccess;
}
"""
FAKE_RUN = """
import json, sys
sys.path.insert(0, "."); sys.path.insert(0, "tests")
import test_gpu_cluster as t
g, p, dt_vd, N = t._sim(tuple(json.loads(sys.argv[1])), t.inputs.PREC_MIXED, 1e-8, 29)
print("CTAS", json.dumps(t._clusters(g, dt_vd)), float(abs(g.field(t.ox.FIELD_P)).sum()).hex())
"""


# where the GPU cannot place a cluster, the next smaller one is taken (the query
# is faked: a preloaded library answers it), with the same mixed fields
@pytest.mark.parametrize("shape,kernel,ctas", [((256, 32, 1), "k_solve_cluster", 16), ((512, 128, 1), "k_mg_cluster", 8)])
def test_clusters_that_cannot_be_placed(tmp_path, shape, kernel, ctas):
    lib = _preload(tmp_path, FAKE_OCCUPANCY)
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    seen = []
    for most in (16, ctas // 2, 1):
        r = subprocess.run([sys.executable, "-c", FAKE_RUN, json.dumps(shape)], cwd=root, capture_output=True, text=True,
                           env=dict(os.environ, LD_PRELOAD=lib, FAKE_CLUSTER=str(most)), timeout=300)
        assert r.returncode == 0, r.stderr[-2000:]
        _, rest = r.stdout.split("CTAS ", 1)
        seen.append((json.loads(rest[:rest.index("}") + 1]), rest.split()[-1]))
    assert seen[0][0] == {kernel: ctas} and list(seen[1][0].values()) == [ctas // 2]
    assert list(seen[2][0].values()) == [1]
    assert seen[0][1] == seen[1][1] == seen[2][1]


# every coarsening ratio inside the cluster (cells of several aspect ratios),
# grids taller than wide, one to sixteen CTAs: the kernel and its CTAs on the
# mixed and on the FP64 path (MG: the V-cycle, SOLVE: the whole solve)
MG, SOLVE = "k_mg_cluster", "k_solve_cluster"
LEVELS = [((24, 48, 40), (16, 2, 2), (MG, 8), (MG, 8)),       # (1, 2, 2) above 1024 cells
          ((24, 48, 40), (32, 2, 2), (MG, 8), (MG, 8)),       # (1, 2, 2) below
          ((48, 6, 40), (2, 32, 2), (MG, 2), (MG, 2)),        # (2, 1, 2)
          ((48, 40, 6), (2, 2, 32), (MG, 2), (MG, 2)),        # (2, 2, 1)
          ((256, 5, 6), (2, 32, 32), (MG, 8), (MG, 8)),       # (2, 1, 1), three in a row on the mixed path
          ((6, 256, 5), (32, 2, 32), (MG, 2), (MG, 2)),       # (1, 2, 1)
          ((5, 6, 256), (32, 32, 2), (MG, 2), (MG, 2)),       # (1, 1, 2)
          ((256, 6, 40), (2, 32, 8), (MG, 8), (MG, 8)),
          ((64, 128, 1), (32, 2, 2), (SOLVE, 16), (MG, 8)),   # (1, 2)
          ((128, 64, 1), (2, 32, 2), (MG, 4), (MG, 4)),       # (2, 1)
          ((19, 120, 1), (2, 1.5, 2), (SOLVE, 2), (MG, 2)), ((40, 200, 1), (2, 1.5, 2), (MG, 4), (MG, 4)),
          ((16, 300, 1), (2, 1.5, 2), (MG, 2), (MG, 2)), ((12, 60, 1), (2, 1.5, 2), (SOLVE, 2), (SOLVE, 2)),
          ((3, 90, 1), (2, 1.5, 2), (SOLVE, 2), (SOLVE, 2)), ((1, 100, 1), (2, 1.5, 2), (SOLVE, 1), (SOLVE, 1)),
          ((9, 33, 21), (2, 1.5, 2), (MG, 2), (MG, 2)), ((12, 40, 40), (2, 1.5, 2), (MG, 2), (MG, 2)),
          ((256, 32, 32), (2, 1.5, 2), (MG, 8), (MG, 8)), ((256, 32, 1), (2, 1.5, 2), (SOLVE, 16), (SOLVE, 16)),
          ((129, 16, 1), (2, 1.5, 2), (SOLVE, 16), (SOLVE, 16)), ((240, 80, 9), (2, 2, 16), (MG, 8), (MG, 8))]


# Mixed: against one CTA, the same bits and so the same PCG iterations. FP64:
# against per-level launches down to the level that is solved exactly. The
# V-cycle is the same but for the order of sums, which changes when a solve
# stops only where its residual meets the target to rounding: at most once in
# the nine solves. (A wrong ghost column, transfer or sweep changes every one.)
@pytest.mark.parametrize("prec", [inputs.PREC_MIXED, inputs.PREC_FP64])
@pytest.mark.parametrize("shape,h,mixed_kernel,fp64_kernel", LEVELS)
def test_cluster_vcycle_is_the_launched_one(shape, h, mixed_kernel, fp64_kernel, prec):
    mixed = prec == inputs.PREC_MIXED
    nx, ny, nz = shape
    c = inputs.random_small_case(31 + nx, nx, ny, nz=nz, dim=3 if nz > 1 else 2, solid_frac=0.1,
                                 hx=h[0] * 1e-6, hy=h[1] * 1e-6, hz=h[2] * 1e-6)
    p = dict(c.params, precision=prec, cg_rtol=1e-8 if mixed else 1e-10, conv_mode=inputs.CONV_PRES_RESID, conv_tol=0.0)
    dt_cfl, dt_b, dt_vd, N = ox.oscar_timesteps(p, 0.02)
    out, its = [], []
    for sched in (dict(), dict(cta_global=0) if mixed else dict(cta_global=0, cta_cells=128)):
        g = ox.Oscar(p, c.solid, c.alpha0)
        g.set_schedule(sched)
        g.drag_step(dt_vd)
        g.relax(dt_vd / N, 2)
        its.append(g.stats()["cg_iters_total"])
        out.append([g.field(w) for w in (ox.FIELD_ALPHA, ox.FIELD_P, ox.FIELD_U, ox.FIELD_U + 1)])
        if not sched:
            kernel, ctas = mixed_kernel if mixed else fp64_kernel
            assert _clusters(g, dt_vd) == {kernel: ctas}
        g.close()
    if mixed:
        assert its[0] == its[1]
        for x, y in zip(*out):
            assert np.array_equal(x, y)
    else:
        assert abs(its[0] - its[1]) <= 1


COUNT_STREAMS = r"""
#include <cuda_runtime.h>
#include <dlfcn.h>
#include <stdio.h>
/* streams on which events are recorded */
static cudaStream_t seen[64];
static int n = 0;
int streams_seen(void) { int m = n; n = 0; return m; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
    int q = 0;
    while (q < n && seen[q] != s) ++q;
    if (q == n && n < 64) seen[n++] = s;
    char so[64];
    snprintf(so, sizeof(so), "libcudart.so.%d", CUDART_VERSION / 1000);
    void *f = dlsym(dlopen(so, RTLD_LAZY), "cudaEventRecord");
    return f ? ((cudaError_t(*)(cudaEvent_t, cudaStream_t))f)(e, s) : cudaErrorUnknown;
}
"""
STREAMS_RUN = """
import ctypes, os, sys
sys.path.insert(0, "."); sys.path.insert(0, "tests")
import test_gpu_cluster as t
streams = ctypes.CDLL(os.environ["LD_PRELOAD"]).streams_seen
g, p, dt_vd, N = t._sim((40, 24, 16), t.inputs.PREC_MIXED, 1e-8, 37)
g.profile(True)
streams()
g.drag_step(dt_vd)
n = streams()
g.profile(False)
print("STREAMS", n, len(g.profile_read()))
"""


def test_timed_steps_run_on_one_stream(tmp_path):
    """In-step timing puts an event pair around every launch; the launches of a
    timed step run one after the other on the instance's stream, so that no
    kernel is timed beside another (a graph step builds the multigrid operators
    on a branch)."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", STREAMS_RUN], cwd=root, capture_output=True, text=True,
                       env=dict(os.environ, LD_PRELOAD=_preload(tmp_path, COUNT_STREAMS)), timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    n, kinds = map(int, r.stdout.split("STREAMS ", 1)[1].split())
    assert n == 1 and kinds > 20
