"""Different handles on different host threads (their work on one stream): the launches
of a handle with a small shared-memory window do not take the room from those of
one with a large window, the kernels of both being the same functions."""
import threading

import numpy as np
import pytest
import scipy.sparse as sp

import workloads as W

pytestmark = pytest.mark.gpu


def blocks(n):
    M = sp.kron(sp.identity(n // 2), np.array([[2.0, -1.0], [-1.0, 2.0]])).tocsr()
    M.sort_indices()
    return W.CSR(n, M.indptr.astype(np.int64), M.indices.astype(np.int32), M.data.astype(np.float64))


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_handles_on_two_threads(prec):
    import torch

    from paper_1312_1553_gb300 import _build, nle

    _build.build()
    nle.load_library()
    precision = nle.NLE_MIXED if prec == "mixed" else nle.NLE_FP64
    # slabs of one CTA, as large as one takes and half of that (the same kernel functions), in 2 x 2 blocks so
    # that a call is short
    n = 8 * 512 * (2 if prec == "fp64" else 4)
    large, small = (blocks(m) for m in (n - 100, n // 2 + 100))
    rng = np.random.default_rng(3)
    work, errors = [], []
    for A in (large, small):
        s = nle.Eigensolver(A, dict(precision=precision, trsv_schedule=nle.NLE_SCHED_LEVEL, trsv_rows=4, grid_ctas=1))
        s.factor_ic(3, 0.0)
        g = torch.from_numpy(rng.standard_normal(A.n)).cuda()
        work.append((s, g, s.apply_prec(g)))
    start = threading.Barrier(2)

    def loop(s, g, ref):
        try:
            start.wait()
            for _ in range(3000):
                if not torch.equal(s.apply_prec(g), ref):
                    errors.append("another result")
        except Exception as e:  # reported by the test below
            errors.append(str(e))

    threads = [threading.Thread(target=loop, args=w) for w in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for s, _, _ in work:
        s.close()
    assert not errors, errors[:3]
