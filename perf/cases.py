"""Cases that stand for what users of this framework run, timed as they call it.

A case names an operation of the public interface, a matrix family with its
grid, the precision and the solver's settings:

  op "shift"    (A - theta I) x                      Eigensolver.apply_shifted
  op "prec"     c = P_k g (Algorithm 3.1)            nle_apply_prec
  op "pcg"      one inner solve of a Newton step     nle_pcg
  op "solve"    the leftmost p eigenpairs            Eigensolver.solve
  op "grad"     the adjoint of a solve               Eigensolver.backward
  op "batch"    many problems in one launch          batch_solve
  op "factor"   IC(lfil, tau) of a new matrix        Eigensolver.factor_ic, nle_get_factor
  op "noalloc"  (L L^T)^{-1} g with a given factor   nle_ic_apply_noalloc

Matrix families (the ones of ``workloads``, built here on the GPU so that
inputs are quick to make): "fd3" 7-point diffusion with face coefficients
exp(Gaussian field), "fd2" 5-point diffusion with log-normal cells, "hex"
27-point trilinear stiffness with log-normal elements, "aniso" the constant
5-point Laplacian a = 1, b = 1.7, "graph" grounded geometric graph Laplacians
(average degree 10).
"""
import ctypes
import math

import numpy as np
import torch

from paper_1312_1553_gb300 import nle

# IC(lfil, tau) of each family, its off-diagonal entries per row of A and of
# L (measured on these families) and the workload the setting comes from
FAMILY = {
    "fd3": dict(lfil=10, tau=1e-3, off_a=6, off_l=9.8),
    "fd2": dict(lfil=30, tau=1e-2, off_a=4, off_l=3.8),
    "hex": dict(lfil=20, tau=1e-4, off_a=26, off_l=19.9),
    "aniso": dict(lfil=5, tau=1e-2, off_a=4, off_l=3.8),
    "graph": dict(lfil=30, tau=1e-2, off_a=9.9, off_l=5.6),
}


def listed():
    return [
        # the smallest call: one product with the shifted matrix of a small
        # 2D problem; launches and host work are all of it
        dict(name="shift_fd2_60x70_f64", op="shift", family="fd2", nx=60, ny=70, nz=1, precision="fp64"),
        # the same product at the benchmark's size, mixed precision
        dict(name="shift_fd3_100_mixed", op="shift", family="fd3", nx=100, ny=100, nz=100, precision="mixed"),
        # the preconditioner as a building block in an outer method: a small
        # 2D problem, the default precision, early in a run (two pairs)
        dict(name="prec_fd2_60x70_f64", op="prec", family="fd2", nx=60, ny=70, nz=1, precision="fp64", k=2, m=2),
        # the same at the benchmark's size with a full ring of pairs
        dict(name="prec_fd3_100_mixed", op="prec", family="fd3", nx=100, ny=100, nz=100, precision="mixed", k=5, m=6),
        # a correction equation of the 27-point stiffness class (wide rows of
        # L), default precision, late in a run (ten deflated vectors)
        dict(name="pcg_hex_48_f64", op="pcg", family="hex", nx=48, ny=48, nz=48, precision="fp64", k=5, m=10,
             its=20),
        # a correction equation of the large 2D class: long, thin dependency
        # chains in L
        dict(name="pcg_fd2_600x700_mixed", op="pcg", family="fd2", nx=600, ny=700, nz=1, precision="mixed", k=5,
             m=4, its=20),
        # a whole solve: the benchmark's matrix, its first two eigenpairs
        dict(name="solve_fd3_100_mixed", op="solve", family="fd3", nx=100, ny=100, nz=100, precision="mixed", p=2,
             tol=1e-8),
        # a whole small solve at the default precision and the tight
        # tolerance of the closed-form check, odd sizes
        dict(name="solve_fd2_61x75_f64", op="solve", family="fd2", nx=61, ny=75, nz=1, precision="fp64", p=4,
             tol=1e-10),
        # training through the eigenpairs: the adjoint of a solve
        dict(name="grad_fd2_60x70_f64", op="grad", family="fd2", nx=60, ny=70, nz=1, precision="fp64", p=3,
             tol=1e-8),
        # many small graphs in one launch (the batched form)
        dict(name="batch_graph_48_mixed", op="batch", family="graph", nx=2000, ny=6000, nz=48, precision="mixed",
             p=2, tol=1e-8),
        # set-up of a new matrix: factor, levels, layouts
        dict(name="factor_fd3_64_mixed", op="factor", family="fd3", nx=64, ny=64, nz=64, precision="mixed"),
        # a caller that may not allocate applies a factor of its own
        dict(name="noalloc_fd3_45x50x55", op="noalloc", family="fd3", nx=45, ny=50, nz=55, precision="fp64"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, family, nmin, nmax):
    """A grid of the family with nmin..nmax unknowns, odd sizes among them."""
    n = math.exp(rng.uniform(math.log(nmin), math.log(nmax)))
    if family in ("fd2", "aniso"):
        nx = max(8, int(math.sqrt(n) * rng.uniform(0.7, 1.2)))
        return nx, max(8, int(n / nx)), 1
    if family == "hex":
        m = max(6, int(n ** (1.0 / 3.0)))
        return m, m, m
    nx = max(6, int(n ** (1.0 / 3.0) * rng.uniform(0.8, 1.1)))
    ny = max(6, int(math.sqrt(n / nx) * rng.uniform(0.85, 1.1)))
    return nx, ny, max(6, int(n / (nx * ny)))


def draw(rng):
    op = rng.choice(["shift", "prec", "prec", "pcg", "pcg", "solve", "grad", "batch", "factor", "noalloc"])
    precision = rng.choice(["fp64", "mixed"])
    if op == "batch":
        lo = rng.randrange(1500, 3000)
        return dict(op=op, family="graph", nx=lo, ny=lo + rng.randrange(500, 3500), nz=rng.randrange(8, 48),
                    precision=precision, p=rng.choice([1, 2]), tol=1e-8)
    family = rng.choice(["fd3", "fd2", "hex", "aniso"] if precision == "fp64" else ["fd3", "fd2", "fd3", "aniso"])
    hi = dict(shift=900000, prec=600000, pcg=400000, solve=30000, grad=5000, factor=250000, noalloc=130000)[op]
    if op == "grad" or (op == "solve" and family == "aniso"):
        family = "fd2"  # a constant stencil can have repeated eigenvalues
    if op == "solve" and family == "hex":
        hi = 10000
    if family == "hex":
        hi = min(hi, 110000)
    if op == "noalloc":
        precision = "fp64"
    nx, ny, nz = _grid(rng, family, 1100, hi)
    c = dict(op=op, family=family, nx=nx, ny=ny, nz=nz, precision=precision)
    if op in ("prec", "pcg"):
        c.update(k=rng.randrange(0, 8), m=rng.randrange(1, 11))
    if op == "pcg":
        c.update(its=rng.randrange(5, 21))
    if op in ("solve", "grad"):
        c.update(p=rng.randrange(1, 4), tol=1e-8)
    return c


# ---------------------------------------------------------------------------
# matrices
# ---------------------------------------------------------------------------

class _Matrix:
    """CSR with numpy arrays, as nle.Eigensolver takes it."""

    def __init__(self, rowptr, col, val):
        self.n = len(rowptr) - 1
        self.rowptr, self.col, self.val = rowptr, col, val


def _dev():
    return torch.device("cuda") if torch.cuda.is_available() else torch.device("cpu")


def _randn(seed, stream, *shape):
    """Seeded N(0,1) on the device."""
    gen = torch.Generator(device=_dev())
    gen.manual_seed((seed * 1000003 + stream * 7919 + 17) % (1 << 62))
    return torch.randn(*shape, generator=gen, dtype=torch.float64, device=_dev())


def _stencil(offsets, coefs):
    """CSR of a structured stencil: coefs[t] (nz, ny, nx) couples node c with
    node c + offsets[t]; couplings that leave the grid are dropped."""
    nz, ny, nx = coefs[0].shape
    order = sorted(range(len(offsets)), key=lambda t: (offsets[t][0] * ny + offsets[t][1]) * nx + offsets[t][2])
    dev = coefs[0].device
    z, y, x = torch.meshgrid(torch.arange(nz, device=dev), torch.arange(ny, device=dev), torch.arange(nx, device=dev),
                             indexing="ij")
    node = ((z * ny + y) * nx + x).reshape(-1)
    M, C, V = [], [], []
    for t in order:
        dz, dy, dx = offsets[t]
        ok = (z + dz >= 0) & (z + dz < nz) & (y + dy >= 0) & (y + dy < ny) & (x + dx >= 0) & (x + dx < nx)
        M.append(ok.reshape(-1))
        C.append(node + ((dz * ny + dy) * nx + dx))
        V.append(coefs[t].reshape(-1))
    M, C, V = torch.stack(M, 1), torch.stack(C, 1), torch.stack(V, 1)
    rp = torch.zeros(node.numel() + 1, dtype=torch.int64, device=dev)
    rp[1:] = torch.cumsum(M.sum(1), 0)
    return _Matrix(rp.cpu().numpy(), C[M].to(torch.int32).cpu().numpy(), V[M].cpu().numpy())


def _gaussian_field(shape, corr, seed):
    """Zero-mean, unit-deviation field: white noise smoothed with
    exp(-d^2 / corr^2) along each axis (in place of the grid's ends, mirrored)."""
    g = _randn(seed, 1, *shape)
    for ax, s in enumerate(shape):
        d = torch.arange(s, dtype=torch.float64, device=g.device)
        K = torch.exp(-((d[:, None] - d[None, :]) / corr) ** 2)
        g = torch.movedim(torch.tensordot(K, g, dims=([1], [ax])), 0, ax)
    g = g - g.mean()
    return g / g.std()


def _fd3(nx, ny, nz, seed):
    g = _gaussian_field((nz, ny, nx), 8.0, seed)
    diag = torch.zeros_like(g)
    offsets, coefs = [(0, 0, 0)], [diag]
    for ax in range(3):
        f = torch.exp(0.5 * (g.narrow(ax, 0, g.shape[ax] - 1) + g.narrow(ax, 1, g.shape[ax] - 1)))
        first, last = torch.exp(g.narrow(ax, 0, 1)), torch.exp(g.narrow(ax, g.shape[ax] - 1, 1))
        lo, hi = torch.cat([first, f], ax), torch.cat([f, last], ax)
        diag += lo + hi
        for sign, face in ((-1, lo), (1, hi)):
            o = [0, 0, 0]
            o[ax] = sign
            offsets.append(tuple(o))
            coefs.append(-face)
    return _stencil(offsets, coefs)


def _fd2(nx, ny, seed):
    k = torch.exp(0.5 * _randn(seed, 1, ny, nx))
    fx = 2 * k[:, :-1] * k[:, 1:] / (k[:, :-1] + k[:, 1:])
    fy = 2 * k[:-1] * k[1:] / (k[:-1] + k[1:])
    west, east = torch.cat([k[:, :1], fx], 1), torch.cat([fx, k[:, -1:]], 1)
    south, north = torch.cat([k[:1], fy], 0), torch.cat([fy, k[-1:]], 0)
    diag = west + east + south + north
    return _stencil([(0, 0, 0), (0, 0, -1), (0, 0, 1), (0, -1, 0), (0, 1, 0)],
                    [c[None] for c in (diag, -west, -east, -south, -north)])


def _aniso(nx, ny, seed):
    # the constant stencil a = 1, b = 1.7; the seed scales it (units of length)
    s = 1.0 + 0.5 * (seed % 97) / 97.0
    one = torch.full((1, ny, nx), s, dtype=torch.float64, device=_dev())
    return _stencil([(0, 0, 0), (0, 0, -1), (0, 0, 1), (0, -1, 0), (0, 1, 0)],
                    [5.4 * one, -one, -one, -1.7 * one, -1.7 * one])


def _hex(m, seed):
    kappa = torch.exp(_randn(seed, 1, m + 1, m + 1, m + 1))
    gp = [0.5 - 0.5 / math.sqrt(3.0), 0.5 + 0.5 / math.sqrt(3.0)]
    K = np.zeros((8, 8))
    for x in gp:
        for y in gp:
            for z in gp:
                G = np.zeros((8, 3))
                for a in range(8):
                    c = [(a >> d) & 1 for d in range(3)]
                    f = [t if b else 1.0 - t for b, t in zip(c, (x, y, z))]
                    s = [1.0 if b else -1.0 for b in c]
                    G[a] = [s[0] * f[1] * f[2], f[0] * s[1] * f[2], f[0] * f[1] * s[2]]
                K += 0.125 * G @ G.T
    ne, h = m + 1, 1.0 / (m + 1)
    offsets, coefs = [], []
    for o in range(27):
        d = (o // 9 - 1, o // 3 % 3 - 1, o % 3 - 1)
        c = torch.zeros(m, m, m, dtype=torch.float64, device=kappa.device)
        for a in range(8):
            az, ay, ax = a >> 2 & 1, a >> 1 & 1, a & 1
            b = (az + d[0], ay + d[1], ax + d[2])
            if min(b) < 0 or max(b) > 1:
                continue
            c = c + kappa[1 - az:ne - az, 1 - ay:ne - ay, 1 - ax:ne - ax] * float(
                h * 0.5 * (K[a, b[2] + 2 * b[1] + 4 * b[0]] + K[b[2] + 2 * b[1] + 4 * b[0], a]))
        offsets.append(d)
        coefs.append(c)
    # both copies of a coupling get the value of the lower one
    for t in range(14, 27):
        u, (dz, dy, dx) = 26 - t, offsets[t]
        lower = torch.roll(coefs[u], shifts=(-dz, -dy, -dx), dims=(0, 1, 2))
        coefs[t] = lower
    return _stencil(offsets, coefs)


def _graph(n, seed):
    """L + 1e-3 I of a connected random geometric graph with n nodes: the n
    nodes nearest (in edges) to one node of the largest component."""
    gen = torch.Generator(device=_dev())
    gen.manual_seed(seed)
    n0 = n + n // 16 + 60
    pts = torch.rand(n0, 2, generator=gen, dtype=torch.float64, device=_dev())
    d2 = (pts[:, None, 0] - pts[None, :, 0]) ** 2 + (pts[:, None, 1] - pts[None, :, 1]) ** 2
    a, b = (t.cpu().numpy() for t in torch.nonzero(torch.triu(d2 < 10.0 / (math.pi * n0), 1), as_tuple=True))
    w = torch.rand(len(a), generator=gen, dtype=torch.float64, device=_dev()).cpu().numpy() * 1.5 + 0.5
    lab = np.arange(n0)
    while True:  # component labels: smallest label of the neighbours, then pointer jumping
        new = lab.copy()
        np.minimum.at(new, a, lab[b])
        np.minimum.at(new, b, lab[a])
        new = new[new]
        if np.array_equal(new, lab):
            break
        lab = new
    dist = np.full(n0, n0)
    dist[np.argmax(np.bincount(lab))] = 0  # a component's label is its first node
    front = True
    while front:
        new = dist.copy()
        np.minimum.at(new, a, dist[b] + 1)
        np.minimum.at(new, b, dist[a] + 1)
        new = np.minimum(new, n0)
        front = not np.array_equal(new, dist)
        dist = new
    keep = np.zeros(n0, bool)
    keep[np.argsort(dist, kind="stable")[:n]] = True
    num = np.cumsum(keep) - 1
    e = keep[a] & keep[b]
    a, b, w = num[a[e]], num[b[e]], w[e]
    deg = np.bincount(a, w, n) + np.bincount(b, w, n) + 1e-3
    rows = np.concatenate([a, b, np.arange(n)])
    cols = np.concatenate([b, a, np.arange(n)])
    vals = np.concatenate([-w, -w, deg])
    o = np.lexsort((cols, rows))
    rp = np.zeros(n + 1, np.int64)
    rp[1:] = np.cumsum(np.bincount(rows, minlength=n))
    return _Matrix(rp, cols[o].astype(np.int32), vals[o])


def _matrix(case, seed):
    f = case["family"]
    if f == "fd3":
        return _fd3(case["nx"], case["ny"], case["nz"], seed)
    if f == "fd2":
        return _fd2(case["nx"], case["ny"], seed)
    if f == "hex":
        return _hex(case["nx"], seed)
    return _aniso(case["nx"], case["ny"], seed)


def _graphs(case, seed):
    """nz graphs with sizes spread evenly over nx..ny points."""
    step = (case["ny"] - case["nx"]) / max(1, case["nz"] - 1)
    return [_graph(int(case["nx"] + b * step), seed * 1000 + b) for b in range(case["nz"])]


def _sines(case, m):
    """The m smoothest products of sines on the grid, orthonormal rows."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    top = range(1, 5)
    modes = sorted(((i, j, l) for i in top for j in top for l in (top if nz > 1 else [0])),
                   key=lambda q: ((q[0] / (nx + 1)) ** 2 + (q[1] / (ny + 1)) ** 2 + (q[2] / (nz + 1)) ** 2, q))[:m]
    rows = []
    for i, j, l in modes:
        x, y, z = (torch.sin(torch.arange(1, s + 1, dtype=torch.float64, device=_dev()) * (q * math.pi / (s + 1)))
                   for q, s in ((i, nx), (j, ny), (l, nz)))
        z = z if l else torch.ones(1, dtype=torch.float64, device=_dev())
        v = (z[:, None, None] * y[None, :, None] * x[None, None, :]).reshape(-1)
        rows.append(v / torch.linalg.vector_norm(v))
    return torch.stack(rows)


def _times(A, x):
    """A x in FP64 (inputs only)."""
    rows = torch.from_numpy(np.repeat(np.arange(A.n), np.diff(A.rowptr))).to(x.device)
    prod = torch.from_numpy(A.val).to(x.device) * x[torch.from_numpy(A.col).to(x.device).long()]
    # row sums by differences of a running sum would lose digits: one slot per row
    return torch.zeros_like(x).index_add_(0, rows, prod) if not x.is_cuda else torch.segment_reduce(
        prod, "sum", lengths=torch.from_numpy(np.diff(A.rowptr)).to(x.device))


def _pairs(A, Q, k, seed):
    """k pairs (s, r) with s^T r < 0, r orthogonal to Q: s = -D^{-1} r, as a
    rough correction of each residual."""
    n = A.n
    rows = np.repeat(np.arange(n), np.diff(A.rowptr))
    d = torch.from_numpy(A.val[A.col == rows]).to(_dev())
    R = _randn(seed, 3, k, n)
    R = R - (R @ Q.T) @ Q
    R = R / torch.linalg.vector_norm(R, dim=1, keepdim=True)
    return (-R / d).contiguous(), R.contiguous()


# ---------------------------------------------------------------------------
# prepare / run
# ---------------------------------------------------------------------------

def _options(case):
    o = dict(precision=nle.NLE_MIXED if case["precision"] == "mixed" else nle.NLE_FP64)
    if case["op"] == "pcg":  # a fixed number of inner iterations
        o.update(exit_eigres=0, exit_stagnation=0, tau_pcg=1e-30)
    if case["op"] == "batch":  # as bench.py runs the batched form
        o.update(grid_ctas=4, trsv_schedule=nle.NLE_SCHED_LEVEL)
    return o


def _solver(case, A):
    nle.load_library()
    s = nle.Eigensolver(A, _options(case))
    s.factor_ic(FAMILY[case["family"]]["lfil"], FAMILY[case["family"]]["tau"])
    return s


def _pcg_inputs(case, A, seed):
    """(theta, r, Q, S, R) of an inner solve: Q smooth and orthonormal with
    the iterate u last, r = A u - q(u) u; theta below the spectrum's start so
    that the system is definite for every matrix."""
    Q = _sines(case, case["m"])
    u = Q[-1]
    Au = _times(A, u)
    q = float(u @ Au)
    S, R = _pairs(A, Q, case["k"], seed)
    Q0 = Q[0]
    theta = 0.3 * min(float(Q0 @ _times(A, Q0)), q)
    return theta, (Au - q * u).contiguous(), Q, S, R


def _parts(F, n, dev):
    """Strictly lower CSR, strictly upper CSR of the transpose, diagonal."""
    rp, col, val = F["Lrowptr"], F["Lcol"], F["Lval"]
    rows = np.repeat(np.arange(n, dtype=np.int32), np.diff(rp))
    off = col != rows
    lr, lc, lv = rows[off], col[off], val[off]
    o = np.argsort(lc, kind="stable")

    def ptr(ix):
        p = np.zeros(n + 1, np.int32)
        p[1:] = np.cumsum(np.bincount(ix, minlength=n))
        return p

    arrays = (ptr(lr), lc, lv, ptr(lc), lr[o], lv[o], val[~off])
    return [torch.from_numpy(np.ascontiguousarray(a)).to(dev) for a in arrays]


def _p(t):
    return ctypes.c_void_p(t.data_ptr()) if t is not None and t.numel() else None


def prepare(case, seed):
    op = case["op"]
    st = dict(case=case)
    if op == "batch":
        mats = _graphs(case, seed)
        st["solvers"] = [_solver(case, A) for A in mats]
        st["X0"] = [_randn(seed, 100 + b, case["p"], A.n) for b, A in enumerate(mats)]
        return st
    A = _matrix(case, seed)
    if op == "factor":
        nle.load_library()
        st["s"] = nle.Eigensolver(A, _options(case))
        # the caller's arrays for the factor, sized by its bound (lfil entries
        # and the diagonal in every column)
        cap = A.n * (FAMILY[case["family"]]["lfil"] + 1)
        st["L"] = dict(nnz=np.zeros(1, np.int64), rowptr=np.zeros(A.n + 1, np.int64), col=np.zeros(cap, np.int32),
                       val=np.zeros(cap), levL=np.zeros(A.n, np.int32), levU=np.zeros(A.n, np.int32),
                       nlevL=np.zeros(1, np.int64), nlevU=np.zeros(1, np.int64))
        return st
    s = st["s"] = _solver(case, A)
    if op == "shift":
        st["x"] = _randn(seed, 2, A.n)
        st["theta"] = 0.01
    elif op == "prec":
        st["Q"] = _sines(case, case["m"])
        st["S"], st["R"] = _pairs(A, st["Q"], case["k"], seed)
        st["g"] = _randn(seed, 2, A.n)
        st["c"] = torch.empty_like(st["g"])
    elif op == "pcg":
        st["theta"], st["r"], st["Q"], st["S"], st["R"] = _pcg_inputs(case, A, seed)
        st["out"] = torch.empty_like(st["r"])
        st["info"] = nle.nle_pcg_info()
    elif op == "solve":
        st["X0"] = _randn(seed, 2, case["p"], A.n)
    elif op == "grad":
        # a loss of the eigenvalues and of the entries of the eigenvectors
        s.solve(case["p"], case["tol"], 200, 20, _randn(seed, 2, case["p"], A.n), allow_noconv=True)
        st["gl"] = _randn(seed, 4, case["p"])
        st["gv"] = _randn(seed, 5, case["p"], A.n)
    elif op == "noalloc":
        st["parts"] = _parts(s.get_factor(), A.n, _dev())
        st["g"] = _randn(seed, 2, A.n)
        st["c"] = torch.empty_like(st["g"])
        st["stream"] = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    return st


def _ok(rc, h):
    if rc != nle.NLE_OK:
        raise nle.NLEError(rc, nle.nle_last_error(h))


def run(st):
    case = st["case"]
    op = case["op"]
    if op == "batch":
        lams, Vs, _ = nle.batch_solve(st["solvers"], case["p"], case["tol"], 400, 20, st["X0"])
        return dict(lam=torch.stack(lams), V=torch.cat([v.reshape(-1) for v in Vs]))
    s = st["s"]
    if op == "shift":
        return s.apply_shifted(st["theta"], st["x"])
    if op == "prec":
        _ok(nle.nle_apply_prec(s.h, case["k"], _p(st["S"]), _p(st["R"]), case["m"], _p(st["Q"]), _p(st["g"]),
                               _p(st["c"]), 1), s.h)
        return st["c"]
    if op == "pcg":
        _ok(nle.nle_pcg(s.h, st["theta"], 1e-8, case["its"], _p(st["r"]), case["m"], _p(st["Q"]), case["k"],
                        _p(st["S"]), _p(st["R"]), _p(st["out"]), st["info"], 1), s.h)
        return dict(s=st["out"], its=int(st["info"].its))
    if op == "solve":
        lam, V, _ = s.solve(case["p"], case["tol"], 200, 20, st["X0"], allow_noconv=True)
        return dict(lam=lam, V=V)
    if op == "grad":
        return s.backward(st["gl"], st["gv"])
    if op == "factor":
        s.factor_ic(FAMILY[case["family"]]["lfil"], FAMILY[case["family"]]["tau"])
        _ok(nle.nle_get_factor(s.h, *(ctypes.c_void_p(a.ctypes.data) for a in st["L"].values())), s.h)
        return st["L"]
    a = st["parts"]
    _ok(nle.nle_ic_apply_noalloc(s.n, *(_p(t) for t in a), _p(st["g"]), _p(st["c"]), st["stream"]), None)
    return st["c"]


# ---------------------------------------------------------------------------
# the work a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    f = FAMILY[case["family"]]
    w = 8 if case["precision"] == "fp64" else 4
    op = case["op"]
    if op == "batch":
        n = case["nz"] * (case["nx"] + case["ny"]) // 2
    else:
        n = case["nx"] * case["ny"] * case["nz"]
    A = n * (1 + f["off_a"]) * (w + 4)
    L = n * (1 + f["off_l"]) * (w + 4)
    fa, fl = 2.0 * n * (1 + f["off_a"]), 2.0 * n * (1 + f["off_l"])
    V = n * w
    if op == "shift":
        return dict(bytes=A + 2 * n * 8, flops=fa + 2 * n)
    if op == "noalloc":
        return dict(bytes=2 * L + 2 * n * 8, flops=2 * fl)
    if op == "factor":
        # A read, L written by rows and by columns with both level arrays
        return dict(bytes=n * (1 + f["off_a"]) * 12 + n * (1 + f["off_l"]) * 12 + 8 * n, flops=fl * f["off_l"])
    if op == "prec":
        k, m = case["k"], case["m"]
        return dict(bytes=2 * L + n * 8 * (2 + 2 * k + m), flops=2 * fl + n * (8.0 * k + 4 * m))
    if op == "pcg":  # per iteration: A, L and L^T once, 16 + 4 k + 4 m vectors
        k, m, its = case["k"], case["m"], case["its"]
        return dict(bytes=its * (A + 2 * L + (16 + 4 * k + 4 * m) * V) + n * 8 * (2 + 2 * k + m),
                    flops=its * (fa + 2 * fl + n * (20.0 + 8 * k + 8 * m)))
    # iterations of a solve and its adjoint grow with the grid's longest side
    # (measured: DACG and inner PCG iterations per eigenpair)
    side = max(case["nx"], case["ny"], case["nz"]) if op != "batch" else math.sqrt(n / case["nz"])
    its = case["p"] * (10 + 1.5 * side) * (2.0 if op == "grad" else 1.0)
    return dict(bytes=its * (A + 2 * L + 30 * V) + 16 * n * case["p"],
                flops=its * (fa + 2 * fl + 40.0 * n))


# ---------------------------------------------------------------------------
# the same results in 64 bits, in plain numpy
# ---------------------------------------------------------------------------

def _ict(A, lfil, tau):
    """L of IC(lfil, tau), by columns: (rows, values) lists, diagonal first."""
    n, rp = A.n, A.rowptr.tolist()
    ci, va = A.col.tolist(), A.val.tolist()
    rows, vals = [None] * n, [None] * n
    at = [[] for _ in range(n)]  # columns whose next entry is in this row, with its position
    for j in range(n):
        w, nrm2 = {j: 0.0}, 0.0
        for e in range(rp[j], rp[j + 1]):
            nrm2 += va[e] * va[e]
            if ci[e] >= j:
                w[ci[e]] = va[e]
        for k, pos in sorted(at[j]):
            rk, vk = rows[k], vals[k]
            l = vk[pos]
            for t in range(pos, len(rk)):
                w[rk[t]] = w.get(rk[t], 0.0) - vk[t] * l
            if pos + 1 < len(rk):
                at[rk[pos + 1]].append((k, pos + 1))
        at[j] = None
        d = math.sqrt(w.pop(j))
        thr = tau * math.sqrt(nrm2)
        keep = [(i, x / d) for i, x in w.items() if not abs(x / d) < thr]
        if len(keep) > lfil:
            keep = sorted(keep, key=lambda q: (-abs(q[1]), q[0]))[:lfil]
        keep.sort()
        rows[j], vals[j] = [j] + [q[0] for q in keep], [d] + [q[1] for q in keep]
        if keep:
            at[rows[j][1]].append((j, 1))
    return rows, vals


class _Tri:
    """(L L^T)^{-1} in numpy, level by level."""

    def __init__(self, n, rows, vals):
        self.n = n
        col = np.repeat(np.arange(n), [len(r) for r in rows])
        row = np.concatenate([np.asarray(r) for r in rows])
        val = np.concatenate([np.asarray(v) for v in vals])
        dg = row == col
        self.diag = val[dg]
        r, c, v = row[~dg], col[~dg], val[~dg]
        self.passes = []
        for i, j in ((r, c), (c, r)):  # entry (i, j): x_i needs x_j
            lev = np.zeros(n, np.int64)
            o = np.argsort(i, kind="stable")
            il, jl = i[o].tolist(), j[o].tolist()
            seq = range(len(il)) if i is r else range(len(il) - 1, -1, -1)
            lv = lev.tolist()
            for e in seq:
                if lv[jl[e]] + 1 > lv[il[e]]:
                    lv[il[e]] = lv[jl[e]] + 1
            lev = np.asarray(lv)
            o = np.argsort(lev[i], kind="stable")
            cut = np.searchsorted(lev[i][o], np.arange(lev.max() + 2))
            ro = np.argsort(lev, kind="stable")
            rcut = np.searchsorted(lev[ro], np.arange(lev.max() + 2))
            self.passes.append((i[o], j[o], v[o], cut, ro, rcut))

    def __call__(self, g):
        x = g
        for i, j, v, cut, ro, rcut in self.passes:
            b, x = x.copy(), np.zeros(self.n)
            for l in range(len(cut) - 1):
                s = slice(cut[l], cut[l + 1])
                if s.stop > s.start:
                    np.subtract.at(b, i[s], v[s] * x[j[s]])
                t = ro[rcut[l]:rcut[l + 1]]
                x[t] = b[t] / self.diag[t]
        return x


def _prec(P0, S, R, Q, g):
    """Algorithm 3.1 and the Gram-Schmidt step, pair by pair."""
    w, a = g.copy(), []
    al = [float(s @ r) for s, r in zip(S, R)]
    for s in range(len(S) - 1, -1, -1):
        a.insert(0, float(S[s] @ w) / al[s])
        w = w - a[0] * R[s]
    c = P0(w)
    for s in range(len(S)):
        b = float(R[s] @ c) / al[s]
        c = c - (a[s] + b) * S[s]
    return c - Q.T @ (Q @ c)


def _dense(A):
    M = np.zeros((A.n, A.n))
    M[np.repeat(np.arange(A.n), np.diff(A.rowptr)), A.col] = A.val
    return M


def _eigs(A, p):
    lam, V = torch.linalg.eigh(torch.from_numpy(_dense(A)))
    lam, V = lam.numpy(), V.numpy()
    return lam, V, V[:, :p].T


def exact(case, seed):
    op, f = case["op"], FAMILY[case["family"]]
    if op == "batch":
        return None  # 48 dense eigenproblems
    n = case["nx"] * case["ny"] * case["nz"]
    if op == "shift":
        A, x = _matrix(case, seed), _randn(seed, 2, n)
        return (_times(A, x) - 0.01 * x).cpu()
    if op in ("solve", "grad"):
        if n > 4700:
            return None  # the dense eigenproblem
        A, p = _matrix(case, seed), case["p"]
        lam, full, V = _eigs(A, p)
        big = np.argmax(np.abs(V), axis=1)
        V = V * np.where(V[np.arange(p), big] < 0, -1.0, 1.0)[:, None]
        if op == "solve":
            return dict(lam=lam[:p].copy(), V=V)
        gl, gv = _randn(seed, 4, p).cpu().numpy(), _randn(seed, 5, p, n).cpu().numpy()
        a, b = np.repeat(np.arange(n), np.diff(A.rowptr)), A.col
        grad = np.zeros(len(b))
        for j in range(p):
            co = full.T @ gv[j]
            gap = lam - lam[j]
            gap[j] = np.inf
            xi = -full @ (co / gap)
            grad += gl[j] * V[j][a] * V[j][b] + xi[a] * V[j][b]
        return grad
    if n * f["off_l"] ** 2 > 6e6:
        return None  # the factor in plain Python
    A = _matrix(case, seed)
    rows, vals = _ict(A, f["lfil"], f["tau"])
    P0 = _Tri(n, rows, vals)
    if op == "noalloc":
        return P0(_randn(seed, 2, n).cpu().numpy())
    if op == "factor":
        col = np.repeat(np.arange(n), [len(r) for r in rows])
        row, val = np.concatenate([np.asarray(r) for r in rows]), np.concatenate([np.asarray(v) for v in vals])
        o = np.lexsort((col, row))
        full = np.zeros(n * (f["lfil"] + 1))
        full[:len(val)] = val[o]
        return dict(val=full)
    if op == "prec":
        Q = _sines(case, case["m"])
        S, R = _pairs(A, Q, case["k"], seed)
        return _prec(P0, S.cpu().numpy(), R.cpu().numpy(), Q.cpu().numpy(), _randn(seed, 2, n).cpu().numpy())
    theta, r, Q, S, R = _pcg_inputs(case, A, seed)
    r, Q, S, R = r.cpu().numpy(), Q.cpu().numpy(), S.cpu().numpy(), R.cpu().numpy()
    a = np.repeat(np.arange(n), np.diff(A.rowptr))

    def J(x):
        y = np.bincount(a, A.val * x[A.col], n) - theta * x
        return y - Q.T @ (Q @ y)

    g = -(r - Q.T @ (Q @ r))
    s = np.zeros(n)
    c = _prec(P0, S, R, Q, g)
    d, gamma = c, float(g @ c)
    for it in range(case["its"]):
        y = J(d)
        alpha = gamma / float(d @ y)
        s, g = s + alpha * d, g - alpha * y
        if it + 1 < case["its"]:
            c = _prec(P0, S, R, Q, g)
            new = float(g @ c)
            d, gamma = c + new / gamma * d, new
    return dict(s=s, its=case["its"])
