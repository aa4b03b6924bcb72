"""Which form of the level schedule a factor takes (nle_stats.trsv_slabs): the
step form for narrow levels, the polled form for FP64 with 2 rows per warp step, for
rows past the step form's entry count and for a window past 192 KB; the chain
schedule has neither.  The polled case with the large window is held to the
oracle, with the bound of test_gpu_long_rows."""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle as O
import workloads as W
from oracle.solver import p0hat
from test_gpu_steps_forms import LEAVES, with_hub

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nle():
    from paper_1312_1553_gb300 import _build, nle

    _build.build()
    nle.load_library()
    return nle


def _solver(nle, A, prec, lfil, tau, **opts):
    s = nle.Eigensolver(A, dict(precision=nle.NLE_MIXED if prec == "mixed" else nle.NLE_FP64, **opts))
    s.factor_ic(lfil, tau)
    return s


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("rows", [4, 2])
@pytest.mark.parametrize("name", ["tridiag", "diff2d5_60x70"])
def test_step_form_runs(nle, name, rows, prec):
    A, lfil, tau = (W.tridiag(2000), 3, 0.0) if name == "tridiag" else (W.workload(name)[0], 30, 1e-2)
    s = _solver(nle, A, prec, lfil, tau, trsv_schedule=nle.NLE_SCHED_LEVEL, trsv_rows=rows)
    assert (s.last_stats()["trsv_slabs"] > 0) == (prec == "mixed" or rows == 4)
    s.close()


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_polled_form_for_long_rows_and_chain(nle, prec):
    A = W.tridiag(2000)
    s = _solver(nle, with_hub(A, LEAVES), prec, 3, 0.0, trsv_schedule=nle.NLE_SCHED_LEVEL, trsv_rows=4)
    assert s.last_stats()["trsv_slabs"] == 0
    s.close()
    s = _solver(nle, A, prec, 3, 0.0, trsv_schedule=nle.NLE_SCHED_CHAIN)
    assert s.last_stats()["trsv_slabs"] == 0
    s.close()


@pytest.mark.parametrize("prec,n", [("fp64", 32500), ("mixed", 65000)])
def test_polled_form_for_a_large_window(nle, prec, n):
    """Four slabs of 64 KB; the last one's halo is nearly all other rows."""
    rng = np.random.default_rng(41)
    i, j = np.repeat(np.arange(n), 4), rng.integers(0, n, 4 * n)
    keep = i != j
    B = sp.coo_matrix((rng.uniform(0.5, 1.0, keep.sum()), (i[keep], j[keep])), shape=(n, n)).tocsr()
    B = B + B.T
    M = (sp.diags(4.0 * np.asarray(B.sum(1)).ravel()) - B).tocsr()
    M.sort_indices()
    A = W.CSR(n, M.indptr.astype(np.int64), M.indices.astype(np.int32), M.data.astype(np.float64))
    s = _solver(nle, A, prec, 8, 0.0, trsv_schedule=nle.NLE_SCHED_LEVEL, trsv_rows=4, grid_ctas=4)
    F = s.get_factor()
    rows = np.repeat(np.arange(n), np.diff(F["Lrowptr"]))
    bsize = (-(-n // 128) * 128 + 15) // 16 * 4
    last = F["Lcol"][rows >= 3 * bsize]
    assert (bsize + len(np.unique(last[last < 3 * bsize]))) * (8 if prec == "fp64" else 4) > 192 * 1024
    assert s.last_stats()["trsv_slabs"] == 0
    g = rng.standard_normal(n)
    ref = p0hat(O.ic_factor(A, 8, 0.0), g)
    c = s.apply_prec(g).cpu().numpy()
    w, eps = np.diff(F["Lrowptr"]).max(), 2.0 ** -53 if prec == "fp64" else 2.0 ** -24
    assert np.abs(c - ref).max() <= 4 * (w + 4) * eps * np.abs(ref).max()
    s.close()
