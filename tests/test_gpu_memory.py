"""A handle holds the layout of the schedule in use, not those of the candidates
the autotuner tried before: the device memory of an automatic handle is that
of one factored for the same schedule and rows alone."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("name", ["diff3d7_64", "graph_60000"])
def test_losing_layouts_are_freed(name, prec):
    import torch

    from paper_1312_1553_gb300 import _build, nle

    _build.build()
    nle.load_library()
    A, lfil, tau = (W.diffusion_3d_7pt(64), 10, 1e-3) if name == "diff3d7_64" else (W.geometric_graph_laplacian(60000, 5), 30,
                                                                                   1e-2)

    def used(**opts):
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        s = nle.Eigensolver(A, dict(precision=nle.NLE_MIXED if prec == "mixed" else nle.NLE_FP64, **opts))
        s.factor_ic(lfil, tau)
        torch.cuda.synchronize()
        got, st = before - torch.cuda.mem_get_info()[0], s.last_stats()
        s.close()
        return got, st

    used()  # kernels and their local memory are loaded
    got, st = used()
    sched = nle.NLE_SCHED_CHAIN if st["trsv_schedule"] == "chain" else nle.NLE_SCHED_LEVEL
    alone, st1 = used(trsv_schedule=sched, trsv_rows=st["trsv_rows"])
    assert st1["trsv_slabs"] == st["trsv_slabs"] and st1["trsv_rows"] == st["trsv_rows"]
    # allocations come in blocks of 2 MB; a layout of these factors is 6 to 100 MB
    assert got <= alone + (4 << 20), (got, alone)
