"""Step form of the triangular solves with long rows (CPU, no GPU).

A step's head holds the entries of a lane in a field of 10 bits.  lfil bounds
the columns of L but not its rows, so one node with many neighbours that is
numbered after them (a hub) gives a row of any length, and a hub numbered
before them a row of L^T of up to lfil entries.  Where the step form is laid
out for such a factor, the layout solves it (by the kernel's rules, see
test_steps_layout); where a lane's entries do not fit, there are no steps and
the library takes the polled form."""
import numpy as np
import pytest

import workloads as W
from test_steps_layout import run, shim, steps  # noqa: F401 (shim is a fixture)

LFIL, TAU = 10000, 0.003


def hub_matrix(r, first):
    """A hub with r neighbours, numbered before (first) or after them, and a
    tridiagonal part of 40 rows behind.  The row of L (of L^T, hub first) has
    r entries; fill between the neighbours is below TAU."""
    import scipy.sparse as sp

    n = r + 41
    hub, leaves = (0, np.arange(1, r + 1)) if first else (r, np.arange(r))
    band = np.arange(r + 1, n)
    d = np.full(n, 4.0)
    if first:
        d[leaves] = r  # column of the hub: 1/2 against TAU sqrt(r); fill 1/(4 sqrt(r)) against TAU r
    else:
        d[hub] = r
    i = np.concatenate([np.full(r, hub), leaves, band[1:], band[:-1], np.arange(n)])
    j = np.concatenate([leaves, np.full(r, hub), band[:-1], band[1:], np.arange(n)])
    M = sp.coo_matrix((np.concatenate([np.full(2 * r + 2 * len(band) - 2, -1.0), d]), (i, j))).tocsr()
    M.sort_indices()
    return W.CSR(n, M.indptr.astype(np.int64), M.indices.astype(np.int32), M.data.astype(np.float64))


@pytest.mark.parametrize("first", [False, True])
@pytest.mark.parametrize("dbl,lpr", [(False, 1), (False, 2), (True, 4)])
@pytest.mark.parametrize("lane", [24, 1023, 1023.25, 1024, 1025, 2048])
def test_long_rows(shim, lane, dbl, lpr, first):  # noqa: F811
    import scipy.sparse as sp
    from scipy.sparse.linalg import spsolve_triangular

    import oracle as O

    r = int(np.ceil(lane * lpr))  # entries of the long row: `lane` per lane
    A = hub_matrix(r, first)
    n = A.n
    ic = O.ic_factor(A, LFIL, TAU)
    L = sp.csr_matrix((ic.Lval, ic.Lcol, ic.Lrowptr), shape=(n, n))
    assert np.diff((L.T if first else L).tocsr().indptr).max() == r + 1
    T = L.T.tocsr() if first else L
    npad = (n + 127) // 128 * 128
    rng = W.rng_for(12)
    rhs = rng.standard_normal(n)
    ref = spsolve_triangular(T, rhs, lower=not first)
    # r + 4 roundings of terms whose magnitudes sum to at most |T||x|, divided by the pivot
    eps = 2.0 ** -53 if dbl else 2.0 ** -24
    diag = T.diagonal()
    tol = 2 * (r + 4) * eps * (abs(T) @ np.abs(ref) / diag).max()
    for grid, nwarps in ((3, 12), (2, 3)):
        bsize = (npad + 4 * grid - 1) // (4 * grid) * 4
        G = steps(shim, A, LFIL, TAU, 0, not first, dbl, bsize, 1, lpr, nwarps)
        if not len(G["head"]):
            assert lane > 24  # rows a step keeps in registers are never left to the polled form
            continue
        x, solved = run(G, n, lpr, nwarps, rhs[G["perm"]], rng)
        assert np.all(solved == 1)
        assert np.abs(x[:n] - ref[G["perm"]]).max() <= tol
