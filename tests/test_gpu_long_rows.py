"""Triangular solves of factors with rows far longer than a warp step holds: a
hub with more neighbours than the step form's entry count can state (1,023 a
lane: 1,023, 2,046 or 4,092 in the row), just as many, and fewer.

The matrices are symmetric M-matrices with off-diagonal row sums of a quarter of the
diagonal and the right-hand sides are positive, so the long rows' sums are a
quarter of the solution.  Conditioning and rounding as in test_gpu_steps: 2 (w + 4) eps a
solve times 2, for rows of w entries.  A hub numbered first has the diagonal 4 and its r
neighbours r, so that their fill, 1 / (4 sqrt(r)), is dropped and the hub's column,
1 / 2, is not: the row of L^T sums r / 2 terms of the size of 1 / r."""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle as O
import workloads as W
from oracle.solver import p0hat

pytestmark = pytest.mark.gpu

# name: (nodes of a ring with random chords, neighbours of each hub, hubs numbered first, lfil)
CASES = {
    "star_1023": (0, (1023,), False, 30),
    "star_1024": (0, (1024,), False, 30),
    "star_4200": (0, (4200,), False, 30),
    "star_9000": (0, (9000,), False, 30),
    "star_first_2100": (0, (2100,), True, 3000),
    "hubs": (12000, (700, 1500, 2500, 5000, 9000), False, 30),
}
_made = {}


def _case(name):
    if name not in _made:
        ring, degrees, first, lfil = CASES[name]
        rng = np.random.default_rng(23)
        m = ring or degrees[0]
        i, j = [], []
        if ring:
            i, j = [np.arange(m), np.arange(m)], [(np.arange(m) + 1) % m, rng.integers(0, m, m)]
        for k, d in enumerate(degrees):
            i.append(np.full(d, m + k))
            j.append(rng.choice(m, d, replace=False))
        n = m + len(degrees)
        i, j = np.concatenate(i), np.concatenate(j)
        keep = i != j
        w = rng.uniform(0.5, 1.0, len(i))
        B = sp.coo_matrix((w[keep], (i[keep], j[keep])), shape=(n, n)).tocsr()
        B = B + B.T
        d = 4.0 * np.asarray(B.sum(1)).ravel()
        if first:
            B, d = (B[::-1, ::-1] > 0).astype(np.float64), np.full(n, float(m))
            d[0] = 4.0
        M = (sp.diags(d) - B).tocsr()
        M.sort_indices()
        A = W.CSR(n, M.indptr.astype(np.int64), M.indices.astype(np.int32), M.data.astype(np.float64))
        ic = O.ic_factor(A, lfil, 0.003 if first else 0.0)
        w = int(max(np.diff(ic.Lrowptr).max(), np.bincount(ic.Lcol).max()))
        assert w > max(degrees)
        g = rng.uniform(0.5, 1.5, n)
        _made[name] = (A, g, p0hat(ic, g), w)
    return _made[name]


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("sched,rows", [("auto", 0), ("level", 4), ("level", 2)])
@pytest.mark.parametrize("name", CASES)
def test_long_rows(name, sched, rows, prec):
    from paper_1312_1553_gb300 import _build, nle

    _build.build()
    nle.load_library()
    A, g, ref, w = _case(name)
    s = nle.Eigensolver(A, dict(precision=nle.NLE_MIXED if prec == "mixed" else nle.NLE_FP64, trsv_rows=rows,
                                trsv_schedule=nle.NLE_SCHED_AUTO if sched == "auto" else nle.NLE_SCHED_LEVEL))
    s.factor_ic(CASES[name][3], 0.003 if CASES[name][2] else 0.0)
    eps = 2.0 ** -53 if prec == "fp64" else 2.0 ** -24
    for _ in range(2):
        c = s.apply_prec(g).cpu().numpy()
        assert np.abs(c - ref).max() <= 4 * (w + 4) * eps * np.abs(ref).max()
    s.close()
