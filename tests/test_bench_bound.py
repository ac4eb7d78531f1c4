"""bench.py says what bounds the dominant kernel kind (no GPU)."""
import bench


def test_bound_names_the_kind_of_limit():
    def table(kind):
        return {kind: (10.0, 4, 4e9), "other": (1.0, 1, 1e9)}

    assert bench.hbm_roofline(table("fp64_residual_pass_a"))["bound"] == "alu"
    assert bench.hbm_roofline(table("inner_pass_ca_rows"))["bound"] == "alu"
    for kind in ("arnoldi_dots", "arnoldi_update", "solution_update", "rhs"):
        r = bench.hbm_roofline(table(kind))
        assert r["bound"] == "hbm" and r["unit"] == "GB/s"
