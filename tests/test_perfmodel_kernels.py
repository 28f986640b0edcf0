"""The operations of the kernels' own formulation (perfmodel.kernel_work) against counts made by walking the
loops on a small shape, and the rooflines that divide them by measured times (no GPU)."""
import pytest

from paper_1807_01151_gb300 import perfmodel as pm


def one_level(dim, p, E, F, form, cls, unit):
    """What level p adds to a cycle."""
    low = pm.kernel_work(dim, p - 1, E, F, form=form)[cls][unit]
    return pm.kernel_work(dim, p, E, F, form=form)[cls][unit] - low


@pytest.mark.parametrize("dim,p", [(2, 1), (2, 3), (3, 2)])
def test_fixed_point_terms_by_loops(dim, p):
    E, F = 7, 19
    s = pm.Shape(dim, p, E, F)
    variables = 4 if dim == 2 else 5
    traces = volume = assembly = 0
    for _e in range(E):
        for _pt in range(s.NF * s.QF):
            traces += variables * s.N                              # U_h at the element's face points
            volume += variables * s.N                              # their fluxes on the modes
            for _pair in range(17 if dim == 2 else 25):
                assembly += s.N * (1 + s.N)
        for _q in range(s.Q):
            volume += variables * s.N + dim * variables * s.N      # U_h, then the gradients
            for _pair in range(17 if dim == 2 else 25):
                assembly += s.N * (dim + s.N)
    residuals = 1 + 2 * 4                                          # of a cycle, two steps of four stages
    assert one_level(dim, p, E, F, 0, "residual_face_flux", "int") == 3 * residuals * traces
    assert one_level(dim, p, E, F, 0, "residual_volume", "int") == 3 * residuals * volume
    assert one_level(dim, p, E, F, 0, "diag_block_assembly", "int") == 3 * 2 * assembly
    assert one_level(dim, p, E, F, 1, "diag_block_assembly", "f32") == 2 * assembly
    assert one_level(dim, p, E, F, 1, "diag_block_assembly", "int") == 0


def test_plane_blocks_and_stages():
    E, N = 5, 15
    assert one_level(2, 4, E, 11, 0, "block_lu", "f64") == pytest.approx(2 * E * (60 ** 3 + 15 ** 3) / 3)
    assert one_level(2, 4, E, 11, 1, "block_lu", "f32") == 2 * E * (60 ** 3 + 15 ** 3)
    assert one_level(2, 4, E, 11, 1, "prk_stage_solve", "bytes") == 8 * E * ((4 * N) ** 2 * 4 + 3 * 75 * 8)
    assert one_level(3, 1, E, 11, 1, "block_lu", "f32") == 2 * E * 20 ** 3


def test_roofline_names_the_slowest_unit():
    import bench
    peaks = {"fp64_tflops": 1.25856, "fp32_tflops": 80.5}
    ops = {"int": 16.3e9, "f64": 0.0, "f32": 80.5e9, "bytes": 6800.0e5}   # 1 ms, 0, 2 ms, 0.1 ms
    r = bench.unit_roofline(ops, 4e-3, peaks, 6800.0)
    assert r["pipe"] == "f32" and r["bound"] == "alu" and r["frac"] == pytest.approx(0.5)
    assert r["achieved"] == pytest.approx(40.25) and r["peak"] == 80.5
    out = bench.unit_rooflines({"block_lu": {"ms_per_cycle": 1.0}, "other": {"ms_per_cycle": 1.0}},
                               {"block_lu": {"int": 0.0, "f64": 0.0, "f32": 0.0, "bytes": 3.4e9}}, peaks, 6800.0)
    assert list(out) == ["block_lu"] and out["block_lu"]["bound"] == "hbm"
    assert out["block_lu"]["frac"] == pytest.approx(0.5) and out["block_lu"]["achieved"] == pytest.approx(3400.0)


def test_measured_kernels_stay_below_their_roofs():
    """128 x 64, p = 4: times of single launches (ncu) against the operations counted for them."""
    E, F = 8192, 16512
    peaks = {"fp64_tflops": 1.25856, "fp32_tflops": 80.5}
    for cls, form, n, us in (("residual_volume", 0, 9, 72.0), ("residual_face_flux", 0, 9, 52.2),
                             ("diag_block_assembly", 0, 2, 1276.0), ("block_lu", 0, 2, 1499.0),
                             ("prk_stage_solve", 0, 8, 142.8)):
        ops = {u: one_level(2, 4, E, F, form, cls, u) / n for u in ("int", "f64", "f32", "bytes")}
        frac = max(pm.unit_times(ops, peaks, 6784.5).values()) / (us * 1e-6)
        assert 0.1 < frac < 1.0, (cls, frac)
