"""Work counts of bench.py for the kernels as they run (no GPU): the stage in nested form and the
element forms on packed integers."""
import pytest

import bench


def test_stage_flops_of_the_nested_form():
    # 47 n1 + 20 n1^2 at n1 = 9
    assert bench.step2r_flops_per_stage() == pytest.approx(4096 * (423 + 1620))


@pytest.mark.parametrize("n1", [4, 9])
def test_element_work(n1):
    NA, tri = n1 * n1, n1 * n1 * (n1 * n1 + 1) // 2 * 8
    faces = 288 * n1 * n1
    state = 72 * n1 * n1 * 8 + 64 * NA
    a0, b0 = bench.element_work(n1, 0, 0, "fp64")
    a1, b1 = bench.element_work(n1, 3, 2, "fp64")
    assert a0 == 4 * NA * NA + faces + 32 * n1**3 and b0 == b1 == 2 * tri + state
    assert a1 - a0 == 5 * (4 * NA * NA + 16 * n1**3)
    # mixed: one limb a product in the inner iterations, four in a sweep's residual
    m0, _ = bench.element_work(n1, 0, 0, "mixed")
    m1, mb = bench.element_work(n1, 3, 2, "mixed", sweeps_u=1.0, sweeps_v=1.0)
    assert m1 - m0 == 5 * NA * NA + 8 * NA * NA and mb == b0
    # inverse: S and both inverses
    assert bench.element_work(n1, 9, 9, "inverse") == (12 * NA * NA + faces, 3 * tri + state)
    with pytest.raises(ValueError):
        bench.element_work(n1, 0, 0, "fp16")


def test_element_roofline_has_no_rate_of_the_equivalent_work(monkeypatch):
    monkeypatch.setattr(bench, "hbm_peak_gbs", lambda: (8000.0, "test"))
    r = bench.element_roofline(4.75e12, 1e9, 1.0, 3e12, 1e12)
    assert r["bound"] == "alu" and r["resource"] == "imad" and r["frac"] == pytest.approx(4.75 / bench.IMAD_PEAK_T)
    assert r["equivalent"] == {"fp64_tflops": 3.0, "fp32_tflops": 1.0} and "frac_fp64" not in r
    r = bench.element_roofline(1e9, 4e12, 1.0, 0.0, 0.0)
    assert r["bound"] == "hbm" and r["unit"] == "GB/s" and r["frac"] == pytest.approx(0.5)
