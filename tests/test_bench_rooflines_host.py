"""What the benchmark says of the kernels it has run (CPU, no GPU): the FP64 factorization by the route
its settings take, and no DRAM traffic that was measured on other kernels."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


@pytest.mark.parametrize("S,L,settings,kernel", [
    (594, 150, {}, "k_factor64_flow"), (594, 150, {"panel_width": 8, "factor_ctas": 152}, "k_factor64_flow"),
    (594, 150, {"factor_ctas": 19}, "k_factor64 "), (594, 150, {"panel_width": 16, "factor_ctas": 152}, "k_factor<double, 16>"),
    (594, 150, {"fp64_panel": 1, "panel_width": 8}, "k_factor_pv<8>"), (96, 150, {"panel_width": 8}, "k_inv64"),
    (96, 150, {"factor_ctas": 152}, "k_factor64_flow"), (96, 7, {}, "k_factor64_flow"), (153, 40, {}, "k_factor64_flow")])
def test_fp64_factorization_by_route(S, L, settings, kernel):
    name, flops = bench.fp64_factorization(S, L, settings)
    assert name.startswith(kernel)
    elimination = 2.0 * S ** 3 * L + 3.0 * S * S * (L - 1)
    if kernel != "k_inv64":
        assert flops == elimination


def test_reduction_products_by_hand():
    """Ten layers: five kept at level 0; level 1 of five eliminates two, level 2 of three one, level 3 of
    two one, without a neighbour above.  [P | Q]: 4 + 2 + 1, Schur terms as many, couplings 2 x 2 + 2 x 1 + 0."""
    S, L = 40, 10
    assert bench.fp64_factorization(S, L, {})[1] == 2.0 * S ** 3 * (L + 2 * (4 + 2 + 1) + 4 + 2)


def test_rooflines_report_no_traffic_of_other_kernels():
    ph = {"factor": (80.0, 10), "tc": (40.0, 1000), "leaf": (30.0, 300)}
    one = dict(tf32=900.0, f32=70.0, f64=1.1, kind="derived")
    out = bench.rooflines(dict(phases=ph, steps=10, work=(1e12, 1e9)), 594, 150, one, one)
    out["fp64"] = bench.roofline_fp64(dict(phases=ph, settings={"panel_width": 8, "factor_ctas": 152}), 594, 150, one, one)
    for key in ("tc", "leaf", "fp64"):
        assert out[key]["traffic"] is None and "traffic_source" not in out[key] and out[key]["achieved"] > 0
