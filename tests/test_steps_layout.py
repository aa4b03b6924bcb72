"""Host logic of the step form of the triangular solves (CPU, no GPU).

The library's own plan_steps and build_steps are compiled with g++ through a
small shim and their output is run by the kernel's rules (trsv_steps): the
steps of a solve slab go round-robin to its warps; a step begins when the
barrier of its warp has got the arrivals its head states (of the ends of
steps that name that barrier, or of the start of the step before in the same
level), the halo values it asks for have been copied in the listed order,
and, after a level too wide for a barrier, that level's steps have reported
their end.  Checked: every operand in the window, no value read that is not
there whichever warps are slow, no barrier with arrivals of two uses at once,
no stall, every row solved once, and the result of the substitution with the
same factor; FP64 and FP32, natural and multicolour orderings, both
directions, all lanes per row, one to three slabs per solve slab, one, two,
three and twelve warps."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle as O
import workloads as W

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
MATS = {
    "aniso2d_30x37": (lambda: W.laplacian_2d_aniso(30, 37, 1.0, 1.7), 5, 1e-2),
    "diff3d7_11x9x10": (lambda: W.diffusion_3d_7pt(11, 9, 10, corr_len=3.0), 10, 1e-3),
    "hex27_9": (lambda: W.hex_poisson_27pt(9), 20, 1e-4),
    "rgg700": (lambda: W.geometric_graph_laplacian(700, 5), 30, 1e-2),
    "tridiag33": (lambda: W.tridiag(33), 3, 0.0),
}
REPORT, EARLY, WAIT = 1, 2, 4


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    out = tmp_path_factory.mktemp("shim") / "libstepsshim.so"
    src = [os.path.join(HERE, "steps_shim.cpp"), os.path.join(ROOT, "paper_1312_1553_gb300", "csrc", "nle_setup.cpp")]
    inc = [f"-I{d}" for d in ("/usr/local/cuda/include", os.path.join(ROOT, "include"))]
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-pthread", "-ffp-contract=off", *inc, *src, "-o",
                    str(out)], check=True)
    lib = ctypes.CDLL(str(out))
    lib.shim_steps.argtypes = [ctypes.c_int64, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int,
                               ctypes.c_double, ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_int64,
                               ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_void_p]
    lib.shim_steps_get.argtypes = [ctypes.c_int] + [ctypes.c_void_p] * 9
    return lib


def steps(lib, A, lfil, tau, colors, lower, dbl, bsize, m, lpr, nwarps):
    rp, ci = np.ascontiguousarray(A.rowptr, np.int64), np.ascontiguousarray(A.col, np.int32)
    va = np.ascontiguousarray(A.val, np.float64)
    sz = np.zeros(6, np.int64)
    assert lib.shim_steps(A.n, rp.ctypes.data, ci.ctypes.data, va.ctypes.data, lfil, tau, colors, int(lower), int(dbl),
                          bsize, m, lpr, nwarps, sz.ctypes.data) == 0
    npad, nslab, nstep, nent, nh, hmax = (int(v) for v in sz)
    G = dict(step0=np.zeros(nslab + 1, np.int32), head=np.zeros((nstep, 8), np.int32),
             row=np.zeros((nstep, 32 // lpr), np.int32), opnd=np.zeros(nent, np.int32), val=np.zeros(nent),
             hptr=np.zeros(nslab + 1, np.int32), hpos=np.zeros(nh, np.int32), diag=np.zeros(A.n), perm=np.zeros(A.n, np.int32))
    lib.shim_steps_get(int(dbl), *[a.ctypes.data for a in G.values()])
    G.update(npad=npad, nslab=nslab, hmax=hmax, rows=m * bsize, size=m * bsize + 1 + hmax, w=8 if dbl else 4)
    return G


def run(G, n, lpr, nwarps, rhs, rng):
    """Reads and ends of the steps as separate events, in an order drawn at
    random among those the rules allow."""
    npad, R = G["npad"], G["rows"]
    x, solved, b, d = np.full(npad, np.nan), np.zeros(npad, int), np.zeros(npad), np.ones(npad)
    b[:n], d[:n] = rhs, G["diag"]
    slabs = []
    for s in range(G["nslab"]):
        win = np.full(G["size"], np.nan)
        win[R] = 0.0
        hp = G["hpos"][G["hptr"][s]:G["hptr"][s + 1]]
        assert np.all((hp >= 0) & (hp < n)) and len(hp) <= G["hmax"]
        ns = int(G["step0"][s + 1] - G["step0"][s])
        # phase of every step: 0 not begun, 1 begun (operands read), 2 ended
        slabs.append(dict(s=s, win=win, hp=hp, have=0, ns=ns, phase=np.zeros(ns, int), bar=[[] for _ in range(nwarps)],
                          sums={}))

    def values(S, c):
        assert np.all((c >= 0) & (c < G["w"] * G["size"]) & (c % G["w"] == 0))
        v = S["win"][c // G["w"]]
        assert not np.isnan(v).any(), "a step reads a value that is not there"
        return v

    def arrive(S, bar, threads):
        # the arrivals of one use of a barrier state the same threads, and never more than that use has
        assert all(q == threads for q in S["bar"][bar]) and 32 * (len(S["bar"][bar]) + 1) < threads
        S["bar"][bar].append(threads)

    while True:
        events = []
        for S in slabs:
            while S["have"] < len(S["hp"]) and not np.isnan(x[S["hp"][S["have"]]]):
                S["win"][R + 1 + S["have"]] = x[S["hp"][S["have"]]]
                S["have"] += 1
            ph = S["phase"]
            lo = int(np.argmax(ph < 2)) if (ph < 2).any() else S["ns"]
            for t in range(lo, min(S["ns"], lo + 2 * nwarps)):
                off, sync, shape, need, first, prev = (int(v) for v in G["head"][G["step0"][S["s"]] + t][:6])
                flags = (shape & 0xFFFFFFFF) >> 16
                ok = ph[t] == 1
                if ph[t] == 0 and (t < nwarps or ph[t - nwarps] == 2) and need <= S["have"]:
                    got = S["bar"][t % nwarps]
                    ok = not sync & 1023 or (32 * (len(got) + 1) == sync & 1023 and all(q == sync & 1023 for q in got))
                    ok = ok and not (flags & WAIT and not np.all(ph[prev:first] == 2))
                if ok:
                    events.append((S, t))
        if not events:
            break
        S, t = events[rng.integers(len(events))]
        off, sync, shape = (int(v) & 0xFFFFFFFF for v in G["head"][G["step0"][S["s"]] + t][:3])
        lanes, quads, flags = shape & 63, ((shape >> 6 & 1023) + 3) // 4, shape >> 16
        nr = lanes // lpr
        rl = G["row"][G["step0"][S["s"]] + t]
        assert np.all(rl[nr:] == rl[nr - 1])
        rl = rl[:nr]
        at0 = S["s"] * R + rl
        if S["phase"][t] == 0:
            at = 4 * (off + np.arange(quads)[:, None] * lanes + np.arange(lanes)[None, :])[:, :, None] + np.arange(4)
            assert np.all(G["val"][at].transpose(0, 2, 1).reshape(-1, lanes)[shape >> 6 & 1023:] == 0)
            S["sums"][t] = (G["val"][at] * values(S, G["opnd"][at])).sum(axis=(0, 2)).reshape(nr, lpr).sum(axis=1)
            if sync & 1023:
                S["bar"][t % nwarps] = []
            if flags & EARLY and nwarps > 1:
                arrive(S, (t + 1) % nwarps, 64)
        else:
            x[at0] = (b[at0] - S["sums"].pop(t)) / d[at0]
            S["win"][rl] = x[at0]
            solved[at0] += 1
            for k in range(sync >> 14 & 15):
                w = ((sync >> 10 & 15) + k) % nwarps
                assert w != t % nwarps  # never its own barrier
                arrive(S, w, sync >> 18)
        S["phase"][t] += 1
    assert all(np.all(S["phase"] == 2) for S in slabs), "the solve stalled"
    assert all(not q for S in slabs for q in S["bar"]), "arrivals without a wait"
    return x, solved


@pytest.mark.parametrize("dbl", [True, False])
@pytest.mark.parametrize("colors", [0, 1, 2])
@pytest.mark.parametrize("lower", [True, False])
@pytest.mark.parametrize("name", list(MATS))
def test_steps_solve_and_never_stall(shim, name, lower, colors, dbl):
    import scipy.sparse as sp
    from scipy.sparse.linalg import spsolve_triangular

    build, lfil, tau = MATS[name]
    A = build()
    n = A.n
    npad = (n + 127) // 128 * 128
    B = W.permute(A, W.multicolor_order(A, colors)[0]) if colors else A
    ic = O.ic_factor(B, lfil, tau)
    L = sp.csr_matrix((ic.Lval, ic.Lcol, ic.Lrowptr), shape=(n, n))
    rng = W.rng_for(12)
    rhs = rng.standard_normal(n)
    P0 = W.multicolor_order(A, colors)[0] if colors else np.arange(n)
    ref = np.zeros(n)
    ref[P0] = spsolve_triangular(L if lower else L.T.tocsr(), rhs[P0], lower=lower)
    # FP64: rounding of two substitutions with well-conditioned factors (condition < 1e3); FP32: coefficients rounded
    # to 2^-24, at most 30 of them in a row
    rtol = 1e-10 if dbl else 1e3 * 30 * 2.0 ** -24
    cases = [(7, 1, 1, 12), (6, 3, 2, 2), (1, 1, 1, 1)] + ([(5, 2, 4, 12), (2, 1, 8, 3)] if dbl else [(4, 2, 1, 3)])
    for grid, m, lpr, nwarps in cases:
        bsize = (npad + 4 * grid - 1) // (4 * grid) * 4
        G = steps(shim, A, lfil, tau, colors, lower, dbl, bsize, m, lpr, nwarps)
        x, solved = run(G, n, lpr, nwarps, rhs[G["perm"]], rng)
        assert np.all(solved == 1)
        np.testing.assert_allclose(x[:n], ref[G["perm"]], rtol=rtol, atol=rtol * 1e-2 * np.abs(ref).max())
