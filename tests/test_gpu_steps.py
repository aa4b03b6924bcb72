"""The level schedule of the triangular solves where its step form can go wrong:
one slab and many, levels of one row (slabs share CTAs, every step needs the step
before, values cross slabs one by one) and levels far wider than the warps in
turn, rows at and past the entries a step keeps in registers, one, two and all
solving warps, a window whose halo is as large as its slab.

The matrices are symmetric M-matrices with off-diagonal row sums of a quarter of the
diagonal.  Their Cholesky columns keep that dominance, the solves are
conditioned by (1 + 1/3) / (1 - 1/3) = 2, and a row of w <= 60 entries, its pivot and the
factor's own rounding give at most 2 (w + 4) eps a solve: 2.6e-16 * 128 * 2 < 1e-13 in
FP64, 2e-5 (eps = 6e-8, the forward error entering the backward solve) in mixed
precision."""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle as O
import workloads as W
from oracle.solver import p0hat

pytestmark = pytest.mark.gpu

# name: (n, band offsets, random entries per row, lfil, grid_ctas)
CASES = {
    "few_rows": (7, (1,), 0, 30, 0),
    "line": (40003, (1,), 0, 30, 0),
    "line_3_ctas": (9001, (1, 2), 0, 30, 3),
    "wide_levels": (20001, (), 1, 30, 0),
    "rows_of_8": (4099, tuple(range(1, 9)), 0, 30, 4),
    "rows_of_17": (4099, tuple(range(1, 18)), 0, 30, 4),
    "rows_of_40": (2050, tuple(range(1, 41)), 0, 60, 0),
    "large_window": (16001, (), 2, 6, 2),
}
_made = {}


def _case(name):
    if name not in _made:
        n, band, per, lfil, ctas = CASES[name]
        rng = np.random.default_rng(17)
        i, j = [np.zeros(0, np.int64)], [np.zeros(0, np.int64)]
        for o in band:
            i.append(np.arange(o, n))
            j.append(np.arange(n - o))
        for _ in range(per):
            i.append(np.arange(n))
            j.append(rng.integers(0, n, n))
        i, j = np.concatenate(i), np.concatenate(j)
        keep = i != j
        B = sp.coo_matrix((rng.uniform(0.5, 1.0, keep.sum()), (i[keep], j[keep])), shape=(n, n)).tocsr()
        B = B + B.T
        M = (sp.diags(4.0 * np.maximum(np.asarray(B.sum(1)).ravel(), 0.25)) - B).tocsr()
        M.sort_indices()
        A = W.CSR(n, M.indptr.astype(np.int64), M.indices.astype(np.int32), M.data.astype(np.float64))
        g = rng.standard_normal(n)
        _made[name] = (A, g, p0hat(O.ic_factor(A, lfil, 0.0), g))
    return _made[name]


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("rows,warps", [(4, 1), (4, 2), (4, 16), (2, 16)])
@pytest.mark.parametrize("name", CASES)
def test_level_solves(name, rows, warps, prec):
    from paper_1312_1553_gb300 import _build, nle

    _build.build()
    nle.load_library()
    A, g, ref = _case(name)
    lfil, ctas = CASES[name][3:]
    s = nle.Eigensolver(A, dict(precision=nle.NLE_MIXED if prec == "mixed" else nle.NLE_FP64, trsv_rows=rows,
                                trsv_schedule=nle.NLE_SCHED_LEVEL, trsv_warps=warps, grid_ctas=ctas))
    s.factor_ic(lfil, 0.0)
    for _ in range(2):
        c = s.apply_prec(g).cpu().numpy()
        assert np.abs(c - ref).max() <= (1e-13 if prec == "fp64" else 2e-5) * np.abs(ref).max()
    s.close()
