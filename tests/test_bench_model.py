"""The bench's per-kernel byte models, on CPU."""
import bench
from paper_2105_10576_gb300 import inputs

CASE = inputs.constricted_channel_3d(nx=64, ny=16, nz=16)


def test_kernels_that_mostly_check_have_no_byte_model():
    """k_cg_refine is launched once per PCG iteration and moves the vectors only
    where a trip ends: no rate follows from its mean time per launch."""
    assert bench.kernel_bytes("k_cg_refine<3>", CASE, 4) is None
    rows, _ = bench.kernel_table([("k_cg_refine<3>", 304, 40.0, 2000), ("k_cg_update<float, 4>", 64, 9.0, 2000)], CASE, 4)
    assert {r["kernel"]: r["gbs"] is None for r in rows} == {"k_cg_refine<3>": True, "k_cg_update<float, 4>": False}
