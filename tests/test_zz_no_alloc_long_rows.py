"""nle_ic_apply_noalloc on factors with long rows: hubs around the length from
which a lane takes four entries at a time (512 in a row, columns unsorted), rows of
many more, factors with more than 32 entries a row on average (one row a warp)
and just below, and a column out of place far inside a long row.

Conditioning and rounding as in test_zz_no_alloc_rows: off-diagonal rows of absolute sum
1/4 on a diagonal of 1 to 2, so both solves together err by at most 2 (w + 4) eps / (3/4) of the
largest |x|, w the entries of the longest row."""
import ctypes

import numpy as np
import pytest
import scipy.sparse as sp

pytestmark = pytest.mark.gpu

# n, entries of the rows: {row: entries}, of all other rows
CASES = {
    "hub_511": (700, {600: 511}, 1),
    "hub_513": (701, {600: 513, 601: 514, 699: 600}, 1),
    "hubs_9000": (9100, {9000: 9000, 9001: 9001, 9002: 5, 9099: 8000}, 2),
    "mean_31": (4099, {}, 31),
    "mean_40": (4099, {}, 40),
    "mean_200": (3001, {2999: 2500}, 200),
    "full": (600, {}, 600),
}


def _lower(n, longer, per, rng):
    rows, vals = [], []
    for i in range(n):
        c = rng.permutation(i)[: min(i, longer.get(i, per))] if i else np.zeros(0, np.int64)
        v = rng.uniform(0.5, 1.0, len(c))
        rows.append(c.astype(np.int32))
        vals.append(v * (0.25 / max(v.sum(), 1e-300)) if len(c) else v)
    return rows, vals


def _call(nle, n, rows, vals, urows, uvals, d, g):
    import torch

    def csr(r, v):
        rp = np.concatenate([[0], np.cumsum([len(c) for c in r])]).astype(np.int32)
        return [rp, np.concatenate(r + [np.zeros(1, np.int32)]).astype(np.int32), np.concatenate(v + [np.zeros(1)])]

    dev = [torch.from_numpy(a).cuda() for a in csr(rows, vals) + csr(urows, uvals) + [d, g]]
    c = torch.empty(n, dtype=torch.float64, device="cuda")
    rc = nle.nle_ic_apply_noalloc(n, *(ctypes.c_void_p(t.data_ptr()) for t in dev), ctypes.c_void_p(c.data_ptr()),
                                  ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    return rc, c.cpu().numpy()


@pytest.fixture(scope="module")
def nle():
    from paper_1312_1553_gb300 import _build, nle

    _build.build()
    nle.load_library()
    return nle


@pytest.mark.parametrize("name", CASES)
def test_long_rows(nle, name):
    n, longer, per = CASES[name]
    rng = np.random.default_rng(n + per)
    rows, vals = _lower(n, longer, per, rng)
    # U: a triangle of the same kind, row n - 1 - i with the mirrored columns
    urows, uvals = [n - 1 - rows[n - 1 - i] for i in range(n)], [vals[n - 1 - i] for i in range(n)]
    d = rng.uniform(1.0, 2.0, n)
    g = rng.uniform(0.5, 1.5, n)
    z, x = np.zeros(n), np.zeros(n)
    for i in range(n):
        z[i] = (g[i] - vals[i] @ z[rows[i]]) / d[i]
    for i in range(n - 1, -1, -1):
        x[i] = (z[i] - uvals[i] @ x[urows[i]]) / d[i]
    w = max(len(r) for r in rows)
    for _ in range(2):
        rc, c = _call(nle, n, rows, vals, urows, uvals, d, g)
        assert rc == nle.NLE_OK, nle.nle_last_error(None)
        assert np.abs(c - x).max() <= 2 * (w + 4) * 2.0 ** -53 / 0.75 * np.abs(x).max()


@pytest.mark.parametrize("name,row", [("hub_513", 601), ("mean_200", 2999)])
def test_column_out_of_place_in_a_long_row(nle, name, row):
    n, longer, per = CASES[name]
    rng = np.random.default_rng(3)
    rows, vals = _lower(n, longer, per, rng)
    rows[row] = rows[row].copy()
    rows[row][len(rows[row]) // 2] = row  # on the diagonal
    urows, uvals = [n - 1 - r for r in _lower(n, {}, 1, rng)[0][::-1]], None
    uvals = [np.full(len(r), 0.1) for r in urows]
    rc, _ = _call(nle, n, rows, vals, urows, uvals, np.ones(n), np.ones(n))
    assert rc == nle.NLE_ERR_CSR
