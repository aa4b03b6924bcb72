"""The level schedule takes its step form only where that is the faster one: stencil
factors with narrow levels, but not graphs in a random numbering, whose slabs need several
times their own rows from other slabs (one iteration of a solve, 20,000 nodes: step
form 275 us in FP64 and 302 mixed, polled form 216 and 250), nor the wide levels of a large
FP64 factor or of a multicolour ordering."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

# matrix, lfil, tau, options; step form in FP64, mixed
CASES = {
    "graph_20000": (lambda: W.geometric_graph_laplacian(20000, 5), 30, 1e-2, {}, False, False),
    "graph_20000_3_ctas": (lambda: W.geometric_graph_laplacian(20000, 5), 30, 1e-2, dict(grid_ctas=3), True, True),
    "diff2d5_150x200_distance_2": (lambda: W.diffusion_2d_lognormal(150, 200), 30, 1e-2, dict(ordering=2), False, True),
    "diff2d5_150x200": (lambda: W.diffusion_2d_lognormal(150, 200), 30, 1e-2, {}, True, True),
    "diff3d7_24": (lambda: W.diffusion_3d_7pt(24), 10, 1e-3, {}, True, True),
    "diff3d7_100": (lambda: W.diffusion_3d_7pt(100), 10, 1e-3, {}, False, True),
}


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("name", CASES)
def test_form(name, prec):
    from paper_1312_1553_gb300 import _build, nle

    _build.build()
    nle.load_library()
    build, lfil, tau, opts, *steps = CASES[name]
    s = nle.Eigensolver(build(), dict(precision=nle.NLE_MIXED if prec == "mixed" else nle.NLE_FP64, trsv_rows=4,
                                      trsv_schedule=nle.NLE_SCHED_LEVEL, **opts))
    s.factor_ic(lfil, tau)
    assert (s.last_stats()["trsv_slabs"] > 0) == steps[prec == "mixed"]
    s.close()
