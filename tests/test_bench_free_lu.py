"""The bench's work split of the LU without a pivot search (CPU): its diagonal blocks, solves and trailing
updates add up to the unblocked LU's multiply-adds, and the profile's groups are charged that split when the
search-free kernels ran."""
import pytest

pytest.importorskip("torch")
import bench  # noqa: E402


@pytest.mark.parametrize("n", [4096, 1000, 129, 128, 5, 1])
def test_free_lu_work_adds_up(n):
    w = bench.free_lu_work(n)
    assert sum(w.values()) == pytest.approx(8.0 * sum((n - k - 1) ** 2 + (n - k - 1) for k in range(n)), rel=1e-12)


def test_the_profile_is_charged_what_ran():
    peaks = {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "sm_max_mhz": 2070.0}
    prof = [("panel_lc_kernel", 32, 2.0), ("lu_trsm_kernel", 32, 1.2), ("cgemm_tc_kernel (trailing update)", 31, 1.1)]
    roof, extra = bench.roofline_from_profile(prof, 4096, 65, 2, 2, peaks, "measured")
    w = bench.free_lu_work(4096)
    assert [r["work_per_step"] for r in [roof] + extra["kernels"]] == [w["diag"], w["trsm"], w["trailing"]]
    roof, _ = bench.roofline_from_profile(prof[:1], 4096, 65, 2, 2, peaks, "measured")
    assert roof["work_per_step"] == bench.lu_work(4096)["panel"]
