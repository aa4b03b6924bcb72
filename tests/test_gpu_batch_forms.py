"""A batch of problems of which some take the step form and some the polled form,
of step-form problems alone and of polled ones alone (three builds of the batched
kernel): each problem's result is that of the oracle."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("kinds", ["both", "steps", "polled"])
def test_batch_of_forms(kinds, prec):
    from paper_1312_1553_gb300 import _build, nle
    from test_gpu_steps_forms import LEAVES, with_hub

    _build.build()
    nle.load_library()
    narrow = [W.diffusion_2d_lognormal(24, 31 + i) for i in range(2)]
    hub = [with_hub(W.diffusion_2d_lognormal(20, 23 + i), LEAVES) for i in range(2)]
    mats = (narrow if kinds != "polled" else []) + (hub if kinds != "steps" else [])
    solvers, X0 = [], []
    for i, A in enumerate(mats):
        s = nle.Eigensolver(A, dict(precision=nle.NLE_MIXED if prec == "mixed" else nle.NLE_FP64, grid_ctas=4,
                                    trsv_schedule=nle.NLE_SCHED_LEVEL, trsv_rows=4))
        s.factor_ic(30, 1e-2)
        assert (s.last_stats()["trsv_slabs"] > 0) == any(A is x for x in narrow)
        solvers.append(s)
        X0.append(W.start_vectors(A.n, 2, 50 + i))
    lams, Vs, per = nle.batch_solve(solvers, 2, 1e-8, 100, 20, X0)
    for A, x0, lam, V, st in zip(mats, X0, lams, Vs, per):
        assert st == 0
        lref, _, _ = O.dacg_newton(A, 2, x0, O.OracleOptions(tol=1e-8, lfil=30, tau_ic=1e-2))
        # a residual of 1e-8 leaves an eigenvalue error of 1e-16 over the relative gap; test_gpu_batch's bounds
        np.testing.assert_allclose(lam.cpu().numpy(), lref, rtol=1e-10 if prec == "fp64" else 1e-8)
    for s in solvers:
        s.close()
