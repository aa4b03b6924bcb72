"""The step form and the polled form of the level schedule give the same bits.

A matrix of two parts that do not touch: the part that is compared, and a hub
behind its neighbours.  With all neighbours the hub's row is too long for a
step and the whole factor takes the polled form; with three of them it takes
the step form.  The other rows of the factor, their levels and so their
numbering are the same in both."""
import numpy as np
import pytest
import scipy.sparse as sp

import workloads as W

pytestmark = pytest.mark.gpu
LEAVES = 4200  # more than 4 x 1,023
# matrix, lfil, tau: rows of L of up to 6, 16, 44 and 26 entries
MATS = {
    "diff2d5_31x37": (lambda: W.diffusion_2d_lognormal(31, 37), 30, 1e-2),
    "diff3d7_15": (lambda: W.diffusion_3d_7pt(15, 15, 15, corr_len=4.0), 10, 1e-3),
    "hex27_13": (lambda: W.hex_poisson_27pt(13), 20, 1e-4),
    "rgg3000": (lambda: W.geometric_graph_laplacian(3000, 5), 30, 1e-2),
}


def with_hub(A, neighbours):
    n = A.n + LEAVES + 1
    i = np.full(neighbours, n - 1)
    j = A.n + np.arange(neighbours)
    S = sp.coo_matrix((-np.ones(neighbours), (i - A.n, j - A.n)), shape=(LEAVES + 1, LEAVES + 1))
    d = np.full(LEAVES + 1, 4.0)
    d[-1] = LEAVES
    M = sp.block_diag([A.to_scipy(), S + S.T + sp.diags(d)]).tocsr()
    M.sort_indices()
    return W.CSR(n, M.indptr.astype(np.int64), M.indices.astype(np.int32), M.data.astype(np.float64))


@pytest.mark.parametrize("prec,rows", [("fp64", 4), ("mixed", 4), ("mixed", 2)])
@pytest.mark.parametrize("name", MATS)
def test_forms_give_the_same_bits(name, prec, rows):
    from paper_1312_1553_gb300 import _build, nle

    _build.build()
    nle.load_library()
    build, lfil, tau = MATS[name]
    A = build()
    rng = W.rng_for(31)
    g = rng.standard_normal((2, A.n + LEAVES + 1))
    out = []
    for neighbours in (LEAVES, 3):
        s = nle.Eigensolver(with_hub(A, neighbours), dict(precision=nle.NLE_MIXED if prec == "mixed" else nle.NLE_FP64,
                                                          trsv_schedule=nle.NLE_SCHED_LEVEL, trsv_rows=rows))
        s.factor_ic(lfil, tau)
        assert (s.last_stats()["trsv_slabs"] > 0) == (neighbours == 3)
        out.append(np.stack([s.apply_prec(x).cpu().numpy()[:A.n] for x in g]))
        s.close()
    np.testing.assert_array_equal(out[0], out[1])
    assert np.all(np.isfinite(out[0])) and np.abs(out[0]).max() > 0
