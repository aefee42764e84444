"""The bench's per-kernel byte models, on CPU."""
import os
import re

import bench
from paper_2105_10576_gb300 import inputs

CASE = inputs.constricted_channel_3d(nx=64, ny=16, nz=16)


def test_kernels_that_mostly_check_have_no_byte_model():
    """k_cg_refine is launched once per PCG iteration and moves the vectors only
    where a trip ends: no rate follows from its mean time per launch."""
    assert bench.kernel_bytes("k_cg_refine<3>", CASE, 4) is None
    rows, _ = bench.kernel_table([("k_cg_refine<3>", 304, 40.0, 2000), ("k_cg_update<float, 4>", 64, 9.0, 2000)], CASE, 4)
    assert {r["kernel"]: r["gbs"] is None for r in rows} == {"k_cg_refine<3>": True, "k_cg_update<float, 4>": False}


def test_fine_sweep_name_is_the_launched_kernel():
    """As many template arguments as the kernel has, the inverse diagonal formed
    by the rule of the launch (whose threshold the source states)."""
    csrc = os.path.join(os.path.dirname(os.path.abspath(bench.__file__)), "paper_2105_10576_gb300", "csrc")
    kern = open(os.path.join(csrc, "oscar_kernels.cuh")).read()
    args = re.search(r"template <([^>]*)>\s*__global__ void k_mg_rbgs\(", kern).group(1)
    name = bench.fine_sweep_name(CASE, 4)
    assert name == "k_mg_rbgs<3, float, false, false>" and name.count(",") == args.count(",")
    assert "kStreamBytes = 80e6" in open(os.path.join(csrc, "oscar_solver.cuh")).read()
    big = inputs.constricted_channel_3d(nx=256, ny=128, nz=128)
    assert bench.fine_sweep_name(big, 4) == "k_mg_rbgs<3, float, false, true>"
    assert bench.fine_sweep_name(big, 8) == "k_mg_rbgs<3, double, false, false>"
    n, F = big.solid.size, bench.grid_counts(big)[1]
    assert bench.kernel_bytes(bench.fine_sweep_name(big, 4), big, 4) == n * 8 + F * 4   # x read, half written, half of b
