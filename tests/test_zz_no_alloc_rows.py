"""nle_ic_apply_noalloc at the edges of its row groups: fewer rows than one
warp's group, remainders, one row past a CTA, rows longer than the entries a
lane group has in flight (16) with unsorted columns, a chain where each row
needs the row before, pivots far outside and inside the range of the corrected
quotient.

The factor has a unit-scale diagonal and off-diagonal rows of absolute sum
<= 1/4 of it, so that ||x||_inf <= ||b||_inf / (3/4 min d) and each solve's rounding
error is at most (w + 4) eps / (3/4) relative to the largest |x|, w <= 64 the entries
of a row: two solves 4e-14, tested at 1e-13."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _factor(n, w, rng, chain):
    rows = []
    for i in range(n):
        c = rng.choice(i, size=min(i, w), replace=False) if i else np.zeros(0, np.int64)
        if chain and i and i - 1 not in c:
            c = np.append(c[:max(0, w - 1)], i - 1)
        rng.shuffle(c)
        rows.append(c.astype(np.int32))
    return rows


@pytest.mark.parametrize("n,w,chain,scale", [(1, 0, False, 1.0), (2, 1, True, 1.0), (3, 2, True, 1.0), (5, 4, False, 1.0),
                                             (127, 7, True, 1.0), (129, 16, False, 1.0), (130, 17, True, 1.0),
                                             (300, 64, False, 1.0), (20001, 3, True, 1.0), (257, 8, True, 1e120),
                                             (257, 8, True, 1e-120)])
def test_row_groups(n, w, chain, scale):
    import torch

    from paper_1312_1553_gb300 import _build, nle

    _build.build()
    nle.load_library()
    rng = np.random.default_rng(1000 + n + w)
    rows = _factor(n, w, rng, chain)
    d = rng.uniform(1.0, 2.0, n)
    vals = []
    for c in rows:
        v = rng.standard_normal(len(c))
        vals.append(v * (0.25 / max(1.0, np.abs(v).sum())))
    # U: a triangle of the same kind, row n - 1 - i with the mirrored columns
    urows, uvals = [n - 1 - rows[n - 1 - i] for i in range(n)], [vals[n - 1 - i] for i in range(n)]
    g = rng.standard_normal(n)
    z = np.zeros(n)
    for i in range(n):
        z[i] = (g[i] - (vals[i] * z[rows[i]]).sum()) / d[i]
    x = np.zeros(n)
    for i in range(n - 1, -1, -1):
        x[i] = (z[i] - (uvals[i] * x[urows[i]]).sum()) / d[i]

    def csr(r, v):
        rp = np.concatenate([[0], np.cumsum([len(c) for c in r])]).astype(np.int32)
        cat = np.concatenate(r) if rp[-1] else np.zeros(1, np.int32)
        return [rp, cat.astype(np.int32), (np.concatenate(v) if rp[-1] else np.zeros(1)) * scale]

    dev = [torch.from_numpy(a).cuda() for a in csr(rows, vals) + csr(urows, uvals) + [d * scale, g]]
    c = torch.empty(n, dtype=torch.float64, device="cuda")
    rc = nle.nle_ic_apply_noalloc(n, *(ctypes.c_void_p(t.data_ptr()) for t in dev), ctypes.c_void_p(c.data_ptr()),
                                  ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == nle.NLE_OK, nle.nle_last_error(None)
    want = x / scale / scale
    assert np.abs(c.cpu().numpy() - want).max() <= 1e-13 * np.abs(want).max()
